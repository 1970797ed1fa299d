"""The selection's bucket path (Sec. 3.4) at the sizes and values where it can go wrong,
bit-exact against the oracle's selection on the same float64 b: clusters whose CTAs own no
bucket, buckets and swap lists at the limits beyond which the general path takes the unit
over, and values whose fp32 intervals are degenerate (one value, infinities, signed zeros,
subnormals, ranges wider than fp32)."""
import numpy as np
import pytest
import torch

import oracle
from gpu_harness import device, split_check
from paper_2608_27128_gb300 import twinkv as tk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    oracle.build()
    tk.load()
    torch.cuda.init()


def _check(b, S0, tau):
    U, N = b.shape
    out = tk.twinkv_repair_select(
        torch.from_numpy(b.reshape(1, U, N)).to(device()),
        torch.from_numpy(S0.reshape(1, U, N)).to(device()),
        torch.from_numpy(S0.sum(1).astype(np.int32)).to(device()), threshold=tau)
    h = {k: v.cpu().numpy() for k, v in out.items()}
    h["score_ret"] = b
    assert np.all(h["status"] == 0)
    split_check(h, S0, tau, 4, 64)
    return h


@pytest.mark.parametrize("cluster", [1, 2, 4, 8])
@pytest.mark.parametrize("kind", ["near", "crowded", "wide", "special", "one value"])
def test_values(kind, cluster, monkeypatch):
    monkeypatch.setenv("TWINKV_SELECT_CLUSTER", str(cluster))
    rng = np.random.default_rng([len(kind), cluster])
    U, N, tau = 4, 2053, 0.5
    S0 = (rng.random((U, N)) < np.array([0.5, 0.3, 0.9, 0.05])[:, None]).astype(np.uint8)
    if kind == "near":
        b = np.where(rng.random((U, N)) < 0.3, 1.0 - 4e-4 * rng.random((U, N)),
                     0.3 + 0.05 * rng.standard_normal((U, N)))
    elif kind == "crowded":     # the largest b within 1e-3 of 1, the rest of the donors far off
        b = np.minimum(1.0, np.where(rng.random((U, N)) < 0.3, 1.0 - rng.exponential(1e-4, (U, N)),
                                     0.5 + 0.1 * rng.standard_normal((U, N))))
    elif kind == "wide":
        b = rng.uniform(-1, 1, (U, N)) * 10.0 ** rng.integers(-320, 308, (U, N))
    elif kind == "special":
        b = rng.choice([0.0, -0.0, -1.0, 1.0, np.inf, -np.inf, 5e-324, 1e300, 0.5], (U, N))
        b[:2] = rng.uniform(-1, 1, (2, N))
        b[0, 100], b[0, 101], b[1, 102] = np.inf, -np.inf, 1e300
    else:
        b = np.where(S0 != 0, 0.75, 0.25)
    _check(b, S0, tau)


@pytest.mark.parametrize("cluster", [1, 2])
@pytest.mark.parametrize("equal", [255, 256, 257])
def test_bucket_at_its_limit(equal, cluster, monkeypatch):
    """`equal` orphans and donors share one value inside the part that is swapped."""
    monkeypatch.setenv("TWINKV_SELECT_CLUSTER", str(cluster))
    rng = np.random.default_rng(equal)
    N = 4099
    S0 = np.zeros((1, N), np.uint8)
    S0[0, rng.permutation(N)[: N // 2]] = 1
    b = np.where(S0 != 0, rng.uniform(0.8, 0.9, (1, N)), rng.uniform(0.2, 0.4, (1, N)))
    for side in (0, 1):
        b[0, rng.permutation(np.flatnonzero(S0[0] == side))[:equal]] = 0.91 if side else 0.1
    _check(b, S0, 0.5)


@pytest.mark.parametrize("cluster", [1, 2, 4])
@pytest.mark.parametrize("donors", [1, 3060, 3071, 3072, 3073, 6140, 6150])
def test_swap_list_at_the_capacity(donors, cluster, monkeypatch):
    monkeypatch.setenv("TWINKV_SELECT_CLUSTER", str(cluster))
    rng = np.random.default_rng([donors, cluster])
    N = 13001
    S0 = np.zeros((1, N), np.uint8)
    S0[0, rng.permutation(N)[: 6400]] = 1
    b = np.where(S0 != 0, 0.3, rng.uniform(-0.2, 0.4, (1, N)))
    inner = np.flatnonzero((S0[0] != 0) & (np.arange(N) >= 4) & (np.arange(N) < N - 64))
    b[0, rng.permutation(inner)[:donors]] = rng.uniform(0.6, 1.0, donors)
    h = _check(b, S0, 0.5)
    assert h["nswaps"][0] == donors
