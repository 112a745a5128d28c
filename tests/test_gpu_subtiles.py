"""The FP64 step's sub-tile rule (8 x 8 sub-tiles up to 608 of them, 16 x 16
beyond) on both sides of its line and at one patch, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2403_15435_gb300 import geoflood, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mi,mj,mx", [(1, 1, 32), (19, 2, 32), (13, 3, 32), (1, 1, 16),
                                      (19, 8, 16), (17, 9, 16)])
def test_small_and_large_forests_match_oracle(mi, mj, mx):
    cfg = inputs.Config(mi=mi, mj=mj, mx=mx, xupper=4.0 * mi * mx, yupper=4.0 * mj * mx,
                        drytol=1e-3, manning_n=0.033, dt_initial=0.1)
    dem = inputs.gaussian_sum_dem(cfg, 12, 5, 8.0)

    def ic(x, y, b):
        # wet and dry cells in every patch, flows in both directions
        h = np.maximum(0.0, 3.5 + 1.5 * np.sin(x / 17.0) * np.cos(y / 23.0) - b)
        return h, 2.0 * h * np.cos(y / 30.0), -3.0 * h * np.sin(x / 40.0)
    g = geoflood.Forest(cfg, dem)
    r = oracle.OracleForest(cfg, dem)
    g.set_state(ic)
    r.set_state(ic)
    assert g.step(1e9, 4) == r.step(1e9, 4)
    for a, b in zip(g.read(), r.read()):
        # four steps from equal states: the parity bound of the FP64 path
        assert np.abs(a - b).max() <= 1e-12 * max(1.0, np.abs(b).max())
