"""The audit's inputs for few units come from one kernel (a cluster per unit), for many from
three: the repair of a unit gives the same bits either way, at the edges of the one kernel's
range (a unit of one tile, ragged and odd lengths, the longest it takes and one more; nine
units and one more), with nothing, everything and one position retained."""
import pytest
import torch

from gpu_harness import device
from paper_2608_27128_gb300 import twinkv as tk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("all_", [False, True])
@pytest.mark.parametrize("N", [1, 31, 256, 513, 1535, 1776, 1792, 1793])
def test_one_kernel_equals_three(N, all_, dtype, d):
    g = torch.Generator(device=device()).manual_seed(N + d)
    U = 24                                            # too many units for clusters of 8
    keys = torch.randn(1, U, N, d, generator=g, device=device())
    keys *= torch.exp2(torch.arange(U, device=device()) * 3 - 36.0)[:, None, None]
    keys[0, 3] = 0.0
    keys[0, 1, N // 2:] = keys[0, 1, :N - N // 2].clone()   # exact twins
    keys = keys.to(dtype)
    mask = (torch.rand(1, U, N, generator=g, device=device()) < 0.5).to(torch.uint8)
    mask[0, 4], mask[0, 5], mask[0, 6] = 0, 7, 0
    mask[0, 6, N - 1] = 1
    kw = dict(threshold=0.5, want_all=True) if all_ else dict(threshold=0.5)
    want = tk.twinkv_repair(keys, mask, **kw)
    for a, b in [(0, 1), (1, 8), (8, 17), (14, 24)]:
        got = tk.twinkv_repair(keys[:, a:b].contiguous(), mask[:, a:b].contiguous(), **kw)
        for name in got:
            x, y = got[name], want[name]
            y = y[:, a:b] if y.dim() == 3 and name != "swaps" else y[a:b]
            if name == "swaps":                       # entries past the count are not written
                n = got["nswaps"].clamp(min=0).tolist()   # -1: the mask of 7s is refused
                assert all(torch.equal(x[i, :n[i]], y[i, :n[i]]) for i in range(b - a)), (a, b)
                continue
            if x.dtype == torch.float64:
                x, y = x.view(torch.int64), y.contiguous().view(torch.int64)
            assert torch.equal(x, y), (name, a, b)
