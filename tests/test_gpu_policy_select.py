"""The policy's selection at the edges of its steps and digits: one step of 8192 positions or
several, one digit of 12 bits or two, lengths that are and are not a multiple of 8, counts
that are all alike (the cut falls among equals) and spread; bit-exact against the oracle's
selection on the same counts."""
import numpy as np
import pytest

from paper_2608_27128_gb300 import synth
from test_gpu_policy import _setup, run_policy  # noqa: F401  (_setup is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [0.95, 0.0, 0.15])
@pytest.mark.parametrize("N", [1, 7, 130, 4095, 4096, 8191, 8192, 8193, 16392])
def test_cut(N, tau):
    rng = np.random.default_rng(N)
    keys = synth.f32_to_bf16_bits(rng.standard_normal((4, N, 64)).astype(np.float32))
    budget = [1, N // 3, max(N - 1, 0), min(N, 70)]
    run_policy(keys, 1, 4, tau, budget, rows=[0, N // 2, N - 1])
