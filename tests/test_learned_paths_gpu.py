"""The learned chains on the mma.sync products, whose exchanges run on a stream
of their own beside the next iteration's first layer: every call gives the
same trajectory, for one, two and many iterations, and counts every chain at
every counted iteration."""
import numpy as np
import pytest

import paper_1507_00315_gb300 as sk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("iters,burnin", [(1, 0), (2, 1), (61, 6)])
def test_exchanges_on_their_own_stream(iters, burnin):
    model = sk.Mlp(0, 12, 640, seed=1)
    model.set_gemm(False)
    beta = np.linspace(0.0, 8.0, 32)
    runs = [sk.pt_run(0, 12, beta, 20, iters, burnin, 3, model=model) for _ in range(3)]
    for r in runs:
        for key in ("hist", "acc_move", "acc_swap"):
            assert np.array_equal(r[key], runs[0][key]), key
        assert int(r["hist"].sum()) == 20 * 32 * (iters - burnin)
    assert iters < 3 or int(runs[0]["acc_swap"].sum()) > 0
    model.close()
