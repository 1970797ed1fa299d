"""The audit at d = 128 over so many small units that each CTA pair passes more segments than
the stamp of a published best tells apart (32), with twins in the first units and none in the
later ones, so that a bound left from an earlier segment would drop a later row's maximum."""
import numpy as np
import pytest
import torch

import oracle
from gpu_harness import device, repair_vs_oracle
from paper_2608_27128_gb300 import synth
from paper_2608_27128_gb300 import twinkv as tk

pytestmark = pytest.mark.gpu


def test_more_segments_than_stamps():
    oracle.build()
    tk.load()
    pairs = torch.cuda.get_device_properties(device()).multi_processor_count // 2
    N, d = 300, 128                    # two work items of two segments per unit
    U = 9 * pairs                      # 18 items, 36 segments per pair
    keys = synth.random_keys(3, U, N, d)
    rng = np.random.default_rng(3)
    for u in range(U // 2):
        p = rng.permutation(N).reshape(-1, 2)
        keys[u, p[:, 1]] = keys[u, p[:, 0]]
    S0 = synth.random_masks(4, U, N, N // 2)
    S0[::7] = 0                        # units whose retained segment is empty
    rep, h, a, r = repair_vs_oracle(keys, S0, 1, U, 8, 0.6)
    assert rep.n_fail == 0, rep.notes
