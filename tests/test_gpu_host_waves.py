"""The host path's chunks at lengths whose number of 128-row blocks is odd: the audit works on
256-row items, one per pair of SMs, so a whole wave counts those."""
import math

import pytest
import torch

import oracle
from gpu_harness import device
from paper_2608_27128_gb300 import synth
from paper_2608_27128_gb300 import twinkv as tk
from test_gpu_host import _assert_same, _device_run, _host_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,H,N,d", [(8, 8, 2432, 128), (36, 8, 300, 64), (36, 8, 16300, 128),
                                     (5, 8, 3200, 64), (36, 8, 3900, 64), (16, 8, 8192, 64)])
def test_default_chunk_is_whole_waves_of_items(L, H, N, d):
    pairs = torch.cuda.get_device_properties(device()).multi_processor_count // 2
    items, U = -(-N // 256), L * H
    step = pairs // math.gcd(pairs, items)
    uc = tk.twinkv_host_default_chunk(tk.Shape(L, H, N, d, tk.BF16))
    assert 1 <= uc <= U
    if step <= U:
        assert (uc * items) % pairs == 0
        want = max((U + 7) // 8, (4 << 20) // (N * d * 2))
        assert abs(uc - want) <= step // 2 + 1 or uc == step


def test_odd_number_of_row_blocks():
    oracle.build()
    tk.load()
    L, H, N = 5, 8, 1120                # nine blocks of 128 rows, the last one partial
    keys = synth.random_keys(11, L * H, N, 64)
    S0 = synth.random_masks(12, L * H, N, N // 2)
    d = _device_run(keys, S0, L, H, 0.4, want_all=True)
    h = _host_run(keys, S0, L, H, 0.4, True, 0, True)
    torch.cuda.synchronize()
    _assert_same(h, d)
