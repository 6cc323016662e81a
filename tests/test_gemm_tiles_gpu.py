"""The proposal network's products at the batches where the column tile
changes (a tile of 64, 128 or 256 columns a CTA; 152 SMs: up to 38 row tiles,
39 to 76, more): the logits of a state do not depend on the batch it is in, and
every gradient block is within the bf16 tolerance of the FP64 backward."""
import numpy as np
import pytest

import paper_1507_00315_gb300 as sk
from oracle import mlp_ref
from tests import seeded_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,n", [(0, 6), (1, 12)])
def test_batches_around_the_tile_rule(variant, n):
    d = si.differences(variant, n)
    off, nslot = mlp_ref.move_table(n, d)
    params = [si.bf16_round(p) for p in si.mlp_params(3, 2 * n, 256, int(nslot.sum()))]
    slots = si.random_slots(11, 9856, n, d)
    model = sk.Mlp(variant, n, 9856, seed=1)
    model.set_params(np.concatenate([x.ravel() for x in params]).astype(np.float32))
    first = model.forward(slots[:128].astype(np.uint8))
    zr = mlp_ref.forward(mlp_ref.occupancy(slots[:128], n, d), *params)[-1]
    assert np.abs(first - zr).max() <= 2e-2 * np.abs(zr).max()
    whole = model.forward(slots.astype(np.uint8))
    assert np.array_equal(whole[:128], first)
    for rows in (4864, 4992, 9728):
        z = model.forward(slots[:rows].astype(np.uint8))
        assert np.array_equal(z, whole[:rows]), rows
    for rows in (128, 4864, 4992, 9728, 9856):
        part = slots[:rows]
        _, g = model.loss_grad(part.astype(np.uint8), 1.5)
        model.check()
        mask = mlp_ref.valid_mask(part, n, d)
        target = mlp_ref.target_distribution(part, n, d, 1.5)
        _, grads = mlp_ref.loss_and_grads(mlp_ref.occupancy(part, n, d), *params, mask, target)
        at = 0
        for name in ("W1", "b1", "W2", "b2", "W3", "b3"):
            ref = np.asarray(grads[name]).ravel()
            got = g[at:at + ref.size]
            at += ref.size
            assert np.linalg.norm(got - ref) <= 3e-2 * np.linalg.norm(ref), (rows, name)
    model.close()
