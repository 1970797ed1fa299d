"""Selections (Sec. 3.4) whose units go beyond one load of the bucket path, bit-exact against
the oracle: buckets with hundreds of equal values (inside the swapped part, at its end, in the
protected and the sliced positions), more such values than the path takes, overfull buckets of
several values, and swap lists of several windows, with and without equal values; the same for
the dedup variant, which leaves them to its general path."""
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


def _scores(kind, U, N, rng):
    b = 0.35 + 0.08 * rng.standard_normal((U, N))
    t = rng.random((U, N))
    near = 1.0 - 4e-4 * rng.random((U, N))
    if kind == "duplicates":        # exact copies: b = 1
        return np.where(t < 0.3, 1.0, b)
    if kind == "both ends":         # equal values on both sides, the orphans' at the list's end
        return np.where(t < 0.25, 1.0, np.where(t < 0.6, 0.3, b))
    if kind == "levels":            # a score of a few levels
        return np.round(np.where(t < 0.3, near, b) * 64) / 64
    if kind == "many levels":       # more levels than overfull buckets are kept of
        return np.round(rng.random((U, N)) * 60) / 60
    if kind == "clump":             # an overfull bucket of different values
        return np.where(t < 0.3, near, np.where(t < 0.9, 0.5 + 1e-6 * b, b))
    if kind == "long":              # lists of several windows
        return np.where(t < 0.5, near, b)
    if kind == "long equal":
        return np.where(t < 0.1, 1.0, np.where(t < 0.5, near, np.where(t < 0.7, 0.31, b)))
    return np.where(t < 0.5, 0.0, 1.0) * np.where(rng.random((U, N)) < 0.5, -1.0, 1.0)   # "signs"


KINDS = ["duplicates", "both ends", "levels", "many levels", "clump", "long", "long equal", "signs"]


def _run(b, S0, tau, twins=None):
    U, N = b.shape
    f = lambda a: torch.from_numpy(a.reshape(1, U, N)).to(device())
    args = (f(b),) if twins is None else (f(b), f(twins))
    fn = tk.twinkv_repair_select if twins is None else tk.twinkv_repair_select_dedup
    out = fn(*args, f(S0), torch.from_numpy(S0.sum(1).astype(np.int32)).to(device()), threshold=tau)
    h = {k: v.cpu().numpy() for k, v in out.items()}
    h["score_ret"] = b
    assert np.all(h["status"] == 0)
    return h


def _masks(U, N, rng):
    return (rng.random((U, N)) < np.array([0.5, 0.3, 0.7])[:U, None]).astype(np.uint8)


@pytest.mark.parametrize("cluster", [1, 2, 8])
@pytest.mark.parametrize("N", [2500, 20011])
@pytest.mark.parametrize("kind", KINDS)
def test_select(kind, N, cluster, monkeypatch):
    monkeypatch.setenv("TWINKV_SELECT_CLUSTER", str(cluster))
    rng = np.random.default_rng([KINDS.index(kind), N, cluster])
    b, S0 = _scores(kind, 3, N, rng), _masks(3, N, rng)
    split_check(_run(b, S0, 0.8), S0, 0.8, 4, 64)


@pytest.mark.parametrize("kind", ["duplicates", "levels", "long", "long equal"])
@pytest.mark.parametrize("N", [131072, (1 << 18) + 1])
def test_select_long_units(kind, N):
    """The library's own cluster size; the longer one is beyond the bucket path."""
    rng = np.random.default_rng([KINDS.index(kind), N])
    b, S0 = _scores(kind, 2, N, rng), _masks(2, N, rng)
    split_check(_run(b, S0, 0.8), S0, 0.8, 4, 64)


@pytest.mark.parametrize("N", [2500, 20011])
@pytest.mark.parametrize("kind", KINDS)
def test_select_dedup(kind, N):
    rng = np.random.default_rng([KINDS.index(kind), N, 7])
    b, S0 = _scores(kind, 3, N, rng), _masks(3, N, rng)
    twins = rng.integers(-1, N, (3, N)).astype(np.int32)
    h = _run(b, S0, 0.8, twins)
    r = oracle.repair_dedup(b, twins, S0, 0.8)
    assert np.array_equal(h["nswaps"], r["nswaps"])
    assert np.array_equal(h["mask"].reshape(3, N), r["mask"])
    for u, m in enumerate(r["nswaps"]):
        assert np.array_equal(h["swaps"][u, :m], np.asarray(r["swaps"][u])[:m])
