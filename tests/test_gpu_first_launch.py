"""The first kernel of a call is fully ordered after the caller's kernel before it on the
stream: read from the edges of a captured graph (nothing of the capture is run).  A
programmatic dependent would wait for that kernel's end only, which need not imply the end of
the work before it if the caller launched it the same way."""
import ctypes

import pytest
import torch

from gpu_harness import device
from paper_2608_27128_gb300 import twinkv as tk

pytestmark = pytest.mark.gpu

L, H, N, D = 1, 2, 2100, 128          # beyond the one-kernel prep


def _edges(stream, fn):
    """[(from, to, type)] of fn() captured on the stream, and the graph's root nodes."""
    cu = ctypes.CDLL("libcuda.so.1")
    P, Z = ctypes.c_void_p, ctypes.c_size_t
    cu.cuStreamBeginCapture_v2.argtypes = [P, ctypes.c_int]
    cu.cuStreamEndCapture.argtypes = [P, ctypes.POINTER(P)]
    cu.cuGraphGetRootNodes.argtypes = [P, P, ctypes.POINTER(Z)]
    cu.cuGraphGetEdges_v2.argtypes = [P, P, P, P, ctypes.POINTER(Z)]
    cu.cuGraphDestroy.argtypes = [P]
    g = P()
    assert cu.cuStreamBeginCapture_v2(stream.cuda_stream, 1) == 0    # thread-local mode
    try:
        fn()
    finally:
        rc = cu.cuStreamEndCapture(stream.cuda_stream, ctypes.byref(g))
    assert rc == 0
    n = Z(64)
    roots = (P * 64)()
    assert cu.cuGraphGetRootNodes(g, roots, ctypes.byref(n)) == 0
    roots = list(roots[:n.value])
    n = Z(64)
    a, b, data = (P * 64)(), (P * 64)(), (ctypes.c_uint8 * (8 * 64))()
    assert cu.cuGraphGetEdges_v2(g, a, b, data, ctypes.byref(n)) == 0
    out = [(a[i], b[i], data[8 * i + 2]) for i in range(n.value)]   # 1: programmatic
    cu.cuGraphDestroy(g)
    return out, roots


@pytest.mark.parametrize("call", ["select", "select_dedup", "noalloc", "repair", "repair_dedup",
                                  "repair_small", "redundancy", "symmetric", "policy"])
def test_first_kernel_is_a_plain_launch(call):
    n = 600 if call == "repair_small" else N      # one prep kernel
    keys = torch.randn(L, H, n, D, device=device()).to(torch.bfloat16)
    mask = (torch.arange(n, device=device()) % 2 == 0).to(torch.uint8).repeat(L, H, 1)
    b = torch.rand(L, H, n, dtype=torch.float64, device=device())
    tw = torch.zeros(L, H, n, dtype=torch.int32, device=device())
    budget = torch.full((L * H,), n // 2, dtype=torch.int32, device=device())
    x = torch.zeros(64, device=device())
    fns = {
        "select": lambda **k: tk.twinkv_repair_select(b, mask, budget, **k),
        "select_dedup": lambda **k: tk.twinkv_repair_select_dedup(b, tw, mask, budget, **k),
        "noalloc": lambda **k: tk.twinkv_repair_select_noalloc(b, mask, budget, **k),
        "repair": lambda **k: tk.twinkv_repair(keys, mask, budget, **k),
        "repair_small": lambda **k: tk.twinkv_repair(keys, mask, budget, **k),
        "repair_dedup": lambda **k: tk.twinkv_repair_dedup(keys, mask, budget, **k),
        "redundancy": lambda **k: tk.twinkv_redundancy(keys, **k),
        "symmetric": lambda **k: tk.twinkv_redundancy_symmetric(keys, **k),
        "policy": lambda **k: tk.twinkv_policy(keys, budget, **k),
    }
    kw = {}
    out = fns[call]()                             # first use, and the outputs to keep
    if isinstance(out, dict):
        kw["out"] = out
    else:
        kw["out_score"], kw["out_twin"] = out
    op = {"select": tk.OP_REPAIR_SELECT, "select_dedup": tk.OP_REPAIR_SELECT_DEDUP,
          "noalloc": None, "redundancy": tk.OP_REDUNDANCY,
          "symmetric": tk.OP_REDUNDANCY_SYMMETRIC, "policy": tk.OP_POLICY}.get(call, tk.OP_REPAIR)
    if op is not None:
        kw["ws"] = tk.workspace(tk.shape_of(keys), op, device())
    s = torch.cuda.Stream()
    torch.cuda.synchronize()

    def fn():
        x.add_(1.0)                               # the caller's kernel: the graph's one root
        fns[call](stream=s, **kw)

    with torch.cuda.stream(s):
        x.add_(1.0)
        torch.cuda.synchronize()
        edges, roots = _edges(s, fn)
    assert len(roots) == 1 and len(edges) >= 1
    first = [t for a, _, t in edges if a == roots[0]]
    assert first and all(t == 0 for t in first), edges
    if call in ("repair", "redundancy", "policy"):   # the later ones are dependents
        assert any(t == 1 for _, _, t in edges), edges
