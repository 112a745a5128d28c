"""Checkpoint loads into a context that already holds DEMs and gauges, of the
same sizes (buffers overwritten in place) and of others (replaced), from bytes
and from other buffers: stepping on from the load equals the saved run."""
import struct

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


def test_load_refuses_dem_sizes_whose_byte_count_wraps():
    prob = inputs.radial_dambreak(64, 32, dx=8.0, radius=120.0)
    f = geoflood.Forest(prob.cfg, inputs.gaussian_sum_dem(prob.cfg, 10, 0, 8.0))
    f.set_state(prob.ic)
    f.step(1e9, 3)
    blob = f.save()
    at = blob.index(struct.pack("<dd", 8.0, 8.0)) - 24  # nx, ny, x0, y0, dx, dy
    nx, ny = struct.unpack_from("<ii", blob, at)
    nx2, ny2 = 2 ** 30 + 23170, 2 ** 31 - 46339
    wrapped = nx2 * ny2 * 8 % 2 ** 64  # 537552: a record of that length parses to its end
    assert (nx, ny) == (65, 65) and nx * ny * 8 < wrapped < 2 ** 20
    data = at + 40
    bad = (blob[:at] + struct.pack("<ii", nx2, ny2) + blob[at + 8:data + nx * ny * 8]
           + bytes(wrapped - nx * ny * 8) + blob[data + nx * ny * 8:])
    g = geoflood.Forest(prob.cfg, None)
    with pytest.raises(geoflood.GeoFloodError, match="corrupt DEM"):
        g.load(bad)
    g.load(blob)
    for a, b in zip(g.read(), f.read()):
        assert np.array_equal(a, b)
