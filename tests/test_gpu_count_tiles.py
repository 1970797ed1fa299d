"""The count audit with its column groups on whole tiles in turn (d = 128) or on halves (64):
odd and even numbers of tiles, one to six of them, so that the tile a group starts an item
with changes from item to item.  Equal units have equal counts whatever items came before
them on their pair, and the first ones agree with the oracle."""
import numpy as np
import pytest
import torch

from gpu_harness import device, keys_tensor
from paper_2608_27128_gb300 import synth
from paper_2608_27128_gb300 import twinkv as tk
from test_gpu_policy import _setup, run_policy  # noqa: F401  (_setup is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("N", [1, 200, 257, 513, 769, 1025, 1536])
def test_items_of_any_number_of_tiles(N, d):
    rng = np.random.default_rng([N, d])
    x = rng.standard_normal((2, N, d)).astype(np.float32)
    x[:, N // 2:] = x[:, :N - N // 2] + 0.3 * x[:, N // 2:]        # counts above zero
    keys = synth.f32_to_bf16_bits(x)
    few, _, _ = run_policy(keys, 1, 2, 0.3, N // 2)
    copies = 80                                                     # several items per pair
    out = tk.twinkv_policy(keys_tensor(np.tile(keys, (copies, 1, 1)), copies, 2),
                           torch.full((2 * copies,), N // 2, dtype=torch.int32, device=device()),
                           threshold=0.3)
    many = out["count"].reshape(copies, 2, N).cpu().numpy()
    np.testing.assert_array_equal(many, np.broadcast_to(few, many.shape))
