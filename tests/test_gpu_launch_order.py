"""The launch order that a step leaves for the next one: each launch counts its
entries in counters of its own and clears those of the launch after it.  Calls
of odd and even numbers of steps, with a scenario that stops early, take the
same patches as one call does: bit for bit, every patch once."""
import numpy as np
import pytest

from paper_2403_15435_gb300 import geoflood, inputs

pytestmark = pytest.mark.gpu


def forest(precision, mx, mi, mj, nscen, flags):
    cfg = inputs.Config(mi=mi, mj=mj, mx=mx, xupper=4.0 * mx * mi, yupper=4.0 * mx * mj,
                        drytol=1e-3, manning_n=0.033, dt_initial=0.1, precision=precision, **flags)
    dem = inputs.gaussian_sum_dem(cfg, 12, 5, 8.0)
    g = geoflood.Forest(cfg, dem, num_scenarios=nscen)
    for s in range(nscen):
        if s:
            g.set_topo(dem, s)

        def ic(x, y, b):
            r = np.hypot(x - cfg.xupper / 3.0, y - cfg.yupper / 2.0)
            h = np.where(r < (4 + s) * mx, np.maximum(0.0, 12.0 - b), 0.0)
            return h, 0.0 * h, 0.0 * h
        g.set_state(ic, s)
    return g


def state(g, nscen):
    # (the clipped volume is a sum in the order in which CTAs end)
    return [a for s in range(nscen) for a in g.read(s)] + [
        np.array([g.time(s)[k] for k in ("t", "dt_next", "steps", "rejects", "nclip")])
        for s in range(nscen)]


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("mx,mi,mj,nscen,flags", [
    (16, 9, 7, 1, {}), (32, 19, 9, 1, {}), (32, 5, 4, 3, {}), (16, 6, 5, 1, {"dim_split": 1})])
def test_calls_of_any_length(precision, mx, mi, mj, nscen, flags):
    a = forest(precision, mx, mi, mj, nscen, flags)
    b = forest(precision, mx, mi, mj, nscen, flags)
    a.step(1e9, 36)
    for n in (1, 2, 3, 1, 17, 5, 7):
        b.step(1e9, n)
    for x, y in zip(state(a, nscen), state(b, nscen)):
        assert np.array_equal(x, y)


def test_scenarios_that_wait():
    # a target close by for all, then far: launches in which nobody steps
    a, b = (forest(1, 32, 5, 4, 2, {}) for _ in range(2))
    a.step(3.0, 400)
    b.step(3.0, 400)
    b.step(3.0, 5)
    b.step(3.0, 8)
    a.step(1e9, 19)
    b.step(1e9, 19)
    for x, y in zip(state(a, 2), state(b, 2)):
        assert np.array_equal(x, y)
