"""The training loss's dE masks over the edges of their ranges: the smallest
order, an order whose bins fill two 32-bit words and ones that need a third
(n >= 33), every pair's first and last slot, crowded and empty bins; loss and
dZ-driven gradients against the FP64 reference (the bf16 tolerances of the
gradient tests), and the logits of batches that are not a multiple of 128."""
import numpy as np
import pytest

import paper_1507_00315_gb300 as sk
from oracle import mlp_ref
from tests import seeded_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,n", [(0, 2), (0, 3), (1, 5), (0, 16), (0, 32), (1, 33), (0, 40)])
def test_loss_and_bias_gradient(variant, n):
    d = si.differences(variant, n)
    off, nslot = mlp_ref.move_table(n, d)
    nm = int(nslot.sum())
    params = [si.bf16_round(p) for p in si.mlp_params(3, 2 * n, 256, nm)]
    slots = si.random_slots(11, 256, n, d)
    slots[0] = 0                                             # every pair at its first slot
    slots[1] = [2 * n - dk - 1 for dk in d]                  # and at its last
    model = sk.Mlp(variant, n, 256, seed=1)
    model.set_params(np.concatenate([x.ravel() for x in params]).astype(np.float32))
    loss, g = model.loss_grad(slots.astype(np.uint8), 1.5)
    model.check()
    mask = mlp_ref.valid_mask(slots, n, d)
    target = mlp_ref.target_distribution(slots, n, d, 1.5)
    want, grads = mlp_ref.loss_and_grads(mlp_ref.occupancy(slots, n, d), *params, mask, target)
    assert abs(loss - want) <= 1e-2 * abs(want)
    # b3's gradient is the column sum of dZ: within the bf16 tolerance of the
    # gradient tests (3e-2 of its norm)
    ref = np.asarray(grads["b3"]).ravel()
    assert np.linalg.norm(g[-nm:] - ref) <= 3e-2 * np.linalg.norm(ref)
    z = model.forward(slots[:77].astype(np.uint8))
    zr = mlp_ref.forward(mlp_ref.occupancy(slots[:77], n, d), *params)[-1]
    assert z.shape == (77, nm) and np.abs(z - zr).max() <= 2e-2 * np.abs(zr).max()
    model.close()
