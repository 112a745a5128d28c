"""Checkpoint loads into a context that already holds DEMs and gauges, of the
same sizes (buffers overwritten in place) and of others (replaced), from bytes
and from other buffers: stepping on from the load equals the saved run."""
import numpy as np
import pytest

from paper_2403_15435_gb300 import geoflood, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
def test_loads_replace_or_reuse_what_a_context_holds(prec):
    prob = inputs.radial_dambreak(64, 32, dx=8.0, radius=120.0)
    prob.cfg.precision = prec
    ckpts, ends = [], []
    for spacing, ng in ((8.0, 3), (8.0, 3), (16.0, 5), (16.0, 0)):
        dem = inputs.gaussian_sum_dem(prob.cfg, 10, len(ckpts), spacing)
        f = geoflood.Forest(prob.cfg, dem)
        f.set_state(prob.ic)
        if ng:
            f.set_gauges(np.stack([np.linspace(100.0, 400.0, ng), np.full(ng, 250.0)], 1))
        f.step(1e9, 3)
        ckpts.append(f.save())
        f.step(1e9, 5)
        ends.append([*f.read(), *f.gauges()])
    g = geoflood.Forest(prob.cfg, None)
    for k in (0, 1, 2, 3, 1, 0, 2):
        g.load(ckpts[k] if k % 2 else bytearray(ckpts[k]))
        g.step(1e9, 5)
        for a, b in zip([*g.read(), *g.gauges()], ends[k]):
            assert np.array_equal(a, b)
