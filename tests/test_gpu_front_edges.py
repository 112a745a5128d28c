"""Edges between wet and dry cells in the FP32 step: scattered wet cells over
broken ground (walls, overtopped steps, one-sided fronts; in a whole 32 x 32
tile more of them than its list holds, and a few), at walls and open
boundaries.  Every kernel shape gives the same bits, and one step from equal
states agrees with the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2403_15435_gb300 import geoflood, inputs

pytestmark = pytest.mark.gpu

# per-step bound of the FP32 path; a wall or a limiter that falls the other
# way within FP32 rounding may exceed it in a cell of a thousand
ABS, SWITCHED = 1e-4, 1e-3


def problem(mi, mj, mx, share, bc, **flags):
    cfg = inputs.Config(mi=mi, mj=mj, mx=mx, xupper=2.0 * mi * mx, yupper=2.0 * mj * mx,
                        drytol=1e-3, manning_n=0.033, dt_initial=0.05, precision=1, bc=bc, **flags)
    dem = inputs.gaussian_sum_dem(cfg, mi * mj * mx // 2, 3, 4.0, width=(3.0, 12.0))

    def ic(x, y, b):
        r = np.modf(np.abs(np.sin(x * 12.9898 + y * 78.233) * 43758.5453))[0]
        h = np.where(r < share, 0.05 + 2.0 * r / share, 0.0)
        return h, h * np.cos(y / 7.0), -1.5 * h * np.sin(x / 9.0)
    return cfg, dem, ic


def forest(p):
    f = geoflood.Forest(p[0], p[1])
    f.set_state(p[2])
    return f


@pytest.mark.parametrize("flags", [{}, {"first_order": 1}])
@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 0, 0, 1), (0, 1, 1, 1)])
@pytest.mark.parametrize("share", [0.5, 0.04, 0.97])
def test_every_shape_keeps_every_bit(share, bc, flags):
    p = problem(4, 3, 32, share, bc, **flags)
    out = []
    for variant in range(8):
        f = forest(p)
        f.set_variant(variant)
        f.step(1e9, 5)
        out.append((f.read()[:3], f.last_t))
    for q, t in out[1:]:
        assert t == out[0][1]
        for a, b in zip(q, out[0][0]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("mi,mj,mx", [(17, 9, 32), (2, 3, 32), (5, 4, 16)])
@pytest.mark.parametrize("share,bc", [(0.5, (0, 0, 0, 0)), (0.04, (1, 0, 0, 1)),
                                      (0.97, (0, 1, 1, 1))])
def test_one_step_matches_oracle(mi, mj, mx, share, bc):
    p = problem(mi, mj, mx, share, bc)
    f = forest(p)
    r = oracle.OracleForest(inputs.Config(**{**p[0].__dict__, "precision": 0}), p[1])
    r.set_state(p[2])
    f.step(1e9, 1)
    r.step(1e9, 1)
    for a, b in zip(f.read()[:3], r.read()[:3]):
        assert (np.abs(a - b) > ABS).mean() <= SWITCHED
