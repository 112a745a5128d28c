"""The FP32 step's sub-tile rule (8 x 8 sub-tiles up to 38 patches of 32 x 32,
16 x 16 up to 152, whole tiles beyond) on both sides of its lines, and patches
without water, which share a CTA by sixteen: bit for bit the fixed whole-tile
shape."""
import numpy as np
import pytest

from paper_2403_15435_gb300 import geoflood, inputs

pytestmark = pytest.mark.gpu


def run(variant, mi, mj, flags, ic, nscen=1, steps=12):
    cfg = inputs.Config(mi=mi, mj=mj, mx=32, xupper=128.0 * mi, yupper=128.0 * mj, drytol=1e-3,
                        manning_n=0.033, dt_initial=0.1, precision=1, **flags)
    dem = inputs.gaussian_sum_dem(cfg, 12, 5, 8.0)
    g = geoflood.Forest(cfg, dem, num_scenarios=nscen)
    for s in range(nscen):
        if s:
            g.set_topo(dem, s)
        g.set_state(lambda x, y, b: ic(x, y, b, s), s)
    g.set_variant(variant)
    g.step(1e9, steps)
    return [a for s in range(nscen) for a in g.read(s)], g.last_t, g.last_steps


def same(a, b):
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
    for x, y in zip(a[0], b[0]):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("flags", [{}, {"first_order": 1}, {"no_transverse": 1}])
@pytest.mark.parametrize("mi,mj", [(1, 1), (19, 2), (13, 3), (19, 8), (17, 9)])
def test_rule_keeps_every_bit(mi, mj, flags):
    def ic(x, y, b, s):  # wet and dry cells in every patch, flows in both directions
        h = np.maximum(0.0, 3.5 + 1.5 * np.sin(x / 17.0) * np.cos(y / 23.0) - b)
        return h, 2.0 * h * np.cos(y / 30.0), -3.0 * h * np.sin(x / 40.0)
    same(run(0, mi, mj, flags, ic), run(2, mi, mj, flags, ic))


@pytest.mark.parametrize("mi,mj,nscen", [(3, 11, 1), (17, 9, 1), (18, 18, 2), (19, 17, 3)])
def test_patches_without_water_share_a_cta(mi, mj, nscen):
    def ic(x, y, b, s):  # a column of water that runs out over dry patches; scenario 1 dry
        r = np.hypot(x - 40.0 * mi, y - 70.0 * mj)
        h = np.where((r < 100.0) & (s != 1), np.maximum(0.0, 12.0 - b), 0.0)
        return h, 0.0 * h, 0.0 * h
    a = run(0, mi, mj, {}, ic, nscen, 48)
    same(a, run(2, mi, mj, {}, ic, nscen, 48))
    assert any((h > 0).any() for h in a[0][::4])
