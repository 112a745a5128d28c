"""The inflow boundary where its two equations hand over: the ghost is joined
to the interior by a rarefaction or by a shock as the inflow's velocity at the
interior depth is below or above the interior's, and the GPU decides that by
the difference's sign where it is clear of rounding.  The ghost cells of an
initial fill against the oracle, with that difference zero, within the margin
on both sides of zero, just outside it and far from it.  Newton's steps end
below 1e-14 relative in both, so the depths agree to 1e-13."""
import numpy as np
import pytest

import oracle
from paper_2403_15435_gb300 import geoflood
from test_gpu_inflow import rotate
from test_oracle_inflow import flood

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [0, 3])
@pytest.mark.parametrize("depth", [0.05, 3.0])
@pytest.mark.parametrize("eps", [0.0, 1e-10, -1e-10, 1e-8, -1e-8, 0.01, -0.01])
def test_ghosts_at_the_handover(eps, depth, side):
    prob = rotate(flood(64, 16, hydrograph=((0.0, 6.0), (100.0, 6.0))), side)
    q = 6.0 / 40.0 * (1.0 - eps)  # four 10 m lines; q / h - u = eps q / h

    def ic(x, y, b):
        h = np.full_like(x, depth)
        n = np.full_like(x, q if side in (0, 2) else -q)
        t = np.zeros_like(x)
        return (h, n, t) if side <= 1 else (h, t, n)
    g = geoflood.Forest(prob.cfg, prob.dem)
    r = oracle.OracleForest(prob.cfg, prob.dem)
    g.set_state(ic)
    r.set_state(ic)
    a, b = g.read_tiles(), r.read_tiles()
    assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max()
    # the inflow's ghosts are among them, next to the interior's depth
    ring = b[:, 0][b[:, 1 if side <= 1 else 2] == (6.0 / 40.0 if side in (0, 2) else -6.0 / 40.0)]
    assert len(ring) >= (8 if eps else 0) and np.abs(ring / depth - 1.0).max(initial=0.0) <= 2 * abs(eps)
