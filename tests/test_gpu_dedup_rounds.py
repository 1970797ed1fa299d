"""The dedup repair's walk as rounds over all donors (Sec. 3.4, distinct b values, so that
the bucket path takes the units), bit-exact against the oracle's sequential walk: twin
graphs that take one round, a few, and more than the kernel's limit, twins that are no
donors, stars, and walks that stop at the number of orphans."""
import numpy as np
import pytest
import torch

import oracle
from gpu_harness import device
from paper_2608_27128_gb300 import twinkv as tk
from test_gpu_dedup import split_check_dedup

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    oracle.build()
    tk.load()
    torch.cuda.init()


@pytest.mark.parametrize("N,kept", [(300, 150), (4096, 2048), (6001, 3000), (6500, 3400)])
@pytest.mark.parametrize("graph", ["mutual", "chain", "reverse chain", "ring", "star", "random"])
def test_graphs(graph, N, kept):
    rng = np.random.default_rng([N, len(graph)])
    S0 = np.zeros((2, N), np.uint8)
    b = rng.uniform(0.0, 0.8, (2, N))
    twin = np.full((2, N), -1, np.int32)
    for u in range(2):
        S0[u, rng.permutation(N)[:kept]] = 1
        ret = np.flatnonzero(S0[u])
        b[u, ret] = rng.uniform(0.85, 1.0, kept)
        order = ret[np.argsort(-b[u, ret])]          # by severity, protected ones among them
        if graph == "mutual":
            p = rng.permutation(ret)[: kept // 2 * 2].reshape(-1, 2)
            twin[u, p[:, 0]], twin[u, p[:, 1]] = p[:, 1], p[:, 0]
        elif graph == "chain":
            twin[u, order[1:]] = order[:-1]
        elif graph == "reverse chain":
            twin[u, order[:-1]] = order[1:]
        elif graph == "ring":
            twin[u, order] = np.roll(order, 1)
        elif graph == "star":
            twin[u, ret] = order[kept // 3]
            twin[u, order[kept // 3]] = order[5]
        else:
            twin[u, ret] = rng.choice(N, kept)
        twin[u][twin[u] == np.arange(N)] = -1
    if N == 6001:                                     # fewer orphans than donors
        evicted = np.flatnonzero(S0[1] == 0)
        b[1, evicted[400:]] = 0.9
    out = tk.twinkv_repair_select_dedup(
        torch.from_numpy(b.reshape(1, 2, N)).to(device()),
        torch.from_numpy(twin.reshape(1, 2, N)).to(device()),
        torch.from_numpy(S0.reshape(1, 2, N)).to(device()),
        torch.from_numpy(S0.sum(1).astype(np.int32)).to(device()), threshold=0.85)
    h = {k: v.cpu().numpy() for k, v in out.items()}
    h["score_ret"], h["twin_ret"] = b, twin
    split_check_dedup(h, S0, 0.85, 4, 64)
