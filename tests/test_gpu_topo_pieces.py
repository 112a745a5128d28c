"""Bed averages on both sides of the bed kernel's rule (up to four DEM pieces
per column or row from tables, more cell by cell): against the oracle, and the
two ways against each other where patches that take different ones share
ghost cells."""
import numpy as np
import pytest

import oracle
from paper_2403_15435_gb300 import geoflood, inputs

pytestmark = pytest.mark.gpu


def dem(x0, x1, y0, y1, d, seed):
    nx, ny = int(np.ceil((x1 - x0) / d)) + 1, int(np.ceil((y1 - y0) / d)) + 1
    z = 40.0 + np.random.default_rng(seed).normal(0.0, 3.0, (ny, nx))
    return inputs.Dem(z=z, x0=x0, y0=y0, dx=d, dy=d)


@pytest.mark.parametrize("mx", [16, 32])
@pytest.mark.parametrize("fine", [None, 8.0, 1.0, 0.9])
def test_beds_from_tables_and_cell_by_cell(mx, fine):
    L = 4.0 * mx  # 4 m cells
    cfg = inputs.Config(mi=4, mj=3, mx=mx, xupper=4 * L, yupper=3 * L, drytol=1e-3)
    dems = [dem(-3.7, 4 * L + 9.0, 1.2, 3 * L - 5.0, 9.3, 1)]  # 9.3 m, less than the domain in y
    if fine is not None:  # over a part of the second column of patches
        dems.insert(0, dem(1.2 * L, 1.7 * L, 0.3 * L, 0.8 * L, fine, 2))
    g = geoflood.Forest(cfg, dems)
    r = oracle.OracleForest(cfg, dems)
    tg, tr = g.read_tiles()[:, 3], r.read_tiles()[:, 3]
    # weights and interpolants of up to some forty pieces in FP64
    assert np.abs(tg - tr).max() <= 1e-13 * np.abs(tr).max()
    lev, px, py = g.patch_info()[:3]
    at = {(x, y): tg[k] for k, (x, y) in enumerate(zip(px, py))}
    for (x, y), t in at.items():
        if (x + 1, y) in at:
            assert np.array_equal(t[2:-2, -2:], at[(x + 1, y)][2:-2, 2:4])
            assert np.array_equal(t[2:-2, -4:-2], at[(x + 1, y)][2:-2, :2])
        if (x, y + 1) in at:
            assert np.array_equal(t[-2:, 2:-2], at[(x, y + 1)][2:4, 2:-2])
