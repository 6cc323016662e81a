"""The tempering kernel's two threshold forms against the oracle's
trajectory: 32-bit thresholds (every acceptance possible, equal temperatures
included) and the general form (an acceptance that underflows to 0, a pair
with one slot), odd and even burn-in and iteration counts, one and two warps a
ladder, ladders that leave lanes idle."""
import numpy as np
import pytest

import oracle
import paper_1507_00315_gb300 as sk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,n", [(0, 2), (1, 2), (1, 3), (0, 7), (1, 11)])
@pytest.mark.parametrize("beta", [[0.0, 0.0, 0.0], [0.0, 1.5, 800.0, 2000.0],
                                  list(np.linspace(0.0, 9.0, 33)),
                                  [0.0] * 20 + list(np.linspace(0.0, 1200.0, 30))])
@pytest.mark.parametrize("iters,burnin", [(201, 17), (64, 0)])
def test_trajectory(variant, n, beta, iters, burnin):
    kw = dict(want_final=True, want_trips=True)
    g = sk.pt_run(variant, n, np.array(beta), 3, iters, burnin, 29, **kw)
    o = oracle.pt_run(variant, n, np.array(beta), 3, iters, burnin, 29, **kw)
    for key in ("hist", "acc_move", "acc_swap", "final_slots", "round_trips"):
        assert np.array_equal(g[key], o[key]), key
