"""Performance cases of the library: what its users have it do, through the
public binding (``geoflood.Forest`` and the C entry point for callers that own
their device memory).

Kinds of case:

``uniform``  a forecast window on a grid without refinement: the analysed state
             goes up from pinned host memory, K adaptive steps, the state comes
             back.
``amr``      the same on a refined forest that is kept for the window (patches
             of several levels, level-change ghosts in every step).
``advance``  a run with regridding: resume from a checkpoint, step to a time
             with the criterion checked and the forest regridded on the way,
             read the final forest and state.  One or several scenarios per
             context; plain or learned tags.
``inflow``   an ``advance`` from an inflow hydrograph onto a dry plain.
``tiles``    one FP64 step of independent tiles on caller-owned device buffers.
``grad``     forward and backward pass of the refinement predictor.

States are synthetic mid-flood states (a collapsing column, a reservoir with a
flood tongue, ...) computed here from the seed, so that the inputs do not
depend on the stepping code.  FP32 contexts hold single-precision states; their
results are returned as float32, FP64 contexts' as float64.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2403_15435_gb300 import geoflood, inputs

G = 9.81
DEV = "cuda" if torch.cuda.is_available() else "cpu"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _uniform(name, mi, mj, mx, precision, steps, front, dx=2.0, manning=0.033, drytol=1e-3,
             first_order=0, no_transverse=0, dim_split=0):
    c = dict(kind="uniform", mi=mi, mj=mj, mx=mx, precision=precision, steps=steps, front=front,
             dx=dx, manning=manning, drytol=drytol, first_order=first_order,
             no_transverse=no_transverse, dim_split=dim_split)
    return dict(c, name=name) if name else c


def _amr(name, terrain, mi, mj, mx, minlevel, maxlevel, precision, steps):
    c = dict(kind="amr", terrain=terrain, mi=mi, mj=mj, mx=mx, minlevel=minlevel,
             maxlevel=maxlevel, precision=precision, steps=steps)
    return dict(c, name=name) if name else c


def _advance(name, mi, mj, mx, maxlevel, precision, nscen, learned, regrid, check, t_end):
    c = dict(kind="advance", mi=mi, mj=mj, mx=mx, maxlevel=maxlevel, precision=precision,
             nscen=nscen, learned=learned, regrid=regrid, check=check, t_end=t_end)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a coarse 64 x 64 basin, eight steps (an interactive
        # what-if, a unit of an ensemble driver): launches, copies and waits
        _uniform("basin64_fp64", 2, 2, 32, 0, 8, 0.30, dx=8.0),
        # the 128 x 128 wet-bed validation grid (dx 5 m, no friction), FP64:
        # every cell wet, few patches
        _uniform("wetbed128_fp64", 4, 4, 32, 0, 40, 0.0, dx=5.0, manning=0.0),
        # radial dam break onto a dry bed, 1024 x 1024 cells of 2 m, both
        # precisions: most of the domain still dry, a front moving
        _uniform("radial1024_fp32", 32, 32, 32, 1, 64, 0.34),
        _uniform("radial1024_fp64", 32, 32, 32, 0, 16, 0.34),
        # the 4 km x 2 km valley on levels 2-4 in FP32, reservoir and flood
        # tongue: the library's headline workload between two regrids
        _amr("valley_fp32", "valley", 16, 8, 32, 2, 4, 1, 96),
        # the 17 km x 9 km canyon (17 x 9 blocks) in 16 x 16 patches, FP32: the
        # largest forest
        _amr("canyon16_fp32", "canyon", 17, 9, 16, 1, 5, 1, 64),
        # the 2 km valley as the paper runs it: FP64, plain tags every 4 steps
        _advance("valley2km_fp64", 4, 2, 32, 3, 0, 1, 0, 4, 4, 2.0),
        # the same in FP32 with the learned tagger, regridding every 64 steps
        _advance("valley2km_learned_fp32", 4, 2, 32, 3, 1, 1, 1, 64, 4, 10.0),
        # 16 breach scenarios of it in one context, FP32, plain tags
        _advance("ensemble16_fp32", 4, 2, 32, 3, 1, 16, 0, 8, 8, 8.0),
        # inflow hydrograph over a dry flood plain: a small forest, hundreds of
        # short steps
        dict(name="floodplain_fp32", kind="inflow", mx=32, maxlevel=3, precision=1, peak=20.0,
             t_end=600.0),
        # the step on 256 tiles of a host code that owns its device memory
        dict(name="tiles256_fp64", kind="tiles", npatch=256, mx=32, wet=0.8),
        # one training batch of the refinement predictor, forward and backward
        dict(name="grad1024", kind="grad", n=1024, pos_weight=4.0),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choice(["uniform", "uniform", "amr", "advance", "advance", "inflow", "tiles", "grad"])
    if kind == "uniform":
        mx, prec = rng.choice([16, 32, 32]), rng.choice([0, 1])
        n = logint(1, 1024 if mx == 32 else 2048)
        mi = max(1, min(n, int(round(math.sqrt(n) * rng.uniform(0.6, 1.6)))))
        mj = max(1, n // mi)
        split = rng.choice([0, 0, 0, 0, 1])
        return _uniform(None, mi, mj, mx, prec, rng.randint(4, 16 if prec == 0 else 64),
                        rng.choice([0.0, round(rng.uniform(0.1, 0.45), 2)])
                        if n <= 64 else round(rng.uniform(0.1, 0.34), 2),
                        dx=rng.choice([2.0, 4.0, 5.0]), manning=rng.choice([0.0, 0.02, 0.033, 0.05]),
                        first_order=rng.choice([0, 0, 0, 1]), dim_split=split)
    if kind == "amr":
        prec = rng.choice([0, 1, 1])
        mx = rng.choice([16, 32])
        top = {(0, 32): 2, (0, 16): 3, (1, 32): 4, (1, 16): 4}[(prec, mx)]
        return _amr(None, "valley", rng.randint(5, 16), rng.randint(3, 8), mx, rng.randint(0, 1),
                    rng.randint(2, top), prec, rng.randint(6, 12 if prec == 0 else 64))
    if kind == "advance":
        prec = rng.choice([0, 1, 1])
        learned = rng.choice([0, 1]) if prec else 0
        chk = rng.choice([4, 8])
        return _advance(None, rng.randint(2, 5), rng.randint(1, 3), rng.choice([16, 32]),
                        rng.randint(2, 3), prec, logint(1, 16 if prec else 2), learned,
                        rng.choice([chk, chk, 64]), chk, round(rng.uniform(1.0, 3.0 if prec == 0 else 5.0), 1))
    if kind == "inflow":
        mx = rng.choice([16, 32])  # the inflow's 20 m hold a line of the finest level
        return dict(kind="inflow", mx=mx, maxlevel=rng.randint(32 // mx, 3),
                    precision=rng.choice([0, 1]), peak=round(rng.uniform(5.0, 30.0), 1),
                    t_end=float(rng.randint(200, 600)))
    if kind == "tiles":
        return dict(kind="tiles", npatch=logint(1, 2048), mx=rng.choice([16, 32]),
                    wet=round(rng.uniform(0.2, 1.0), 2))
    return dict(kind="grad", n=logint(64, 4096), pos_weight=round(rng.uniform(1.0, 8.0), 1))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _pinned(shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, pin_memory=DEV == "cuda")


def _smooth(gen, xn, yn, Lx, Ly, count, wl):
    """Sum of `count` seeded plane waves of unit total amplitude on the grid
    (xn, yn), wavelengths around `wl`."""
    k = gen.uniform(0.5, 1.5, count) * 2 * np.pi / wl
    a = gen.uniform(0, 2 * np.pi, count)
    ph = gen.uniform(0, 2 * np.pi, count)
    out = torch.zeros(len(yn), len(xn), dtype=torch.float64, device=DEV)
    X = torch.as_tensor(xn, dtype=torch.float64, device=DEV)[None, :]
    Y = torch.as_tensor(yn, dtype=torch.float64, device=DEV)[:, None]
    for i in range(count):
        out += torch.sin(k[i] * (math.cos(a[i]) * X + math.sin(a[i]) * Y) + ph[i])
    return out / count


def _uniform_input(case, seed):
    """(cfg, nodal bed [ny+1][nx+1], h, hu, hv on the whole grid [ny][nx], dt0):
    seeded rolling terrain with nodes on the cell corners, and a column of
    water that has collapsed to a front radius of `front` times the shorter
    side (0: the whole basin under water, a swell on it)."""
    m, dx = case["mx"], case["dx"]
    nx, ny = case["mi"] * m, case["mj"] * m
    Lx, Ly = nx * dx, ny * dx
    cfl = 0.45 if case["no_transverse"] else 0.9
    cfg = inputs.Config(mi=case["mi"], mj=case["mj"], mx=m, xupper=Lx, yupper=Ly,
                        drytol=case["drytol"], manning_n=case["manning"],
                        cfl_desired=cfl, cfl_max=cfl + 0.05 if cfl < 0.5 else 1.0,
                        tag_depth=case["drytol"], precision=case["precision"],
                        first_order=case["first_order"], no_transverse=case["no_transverse"],
                        dim_split=case["dim_split"])
    gen = np.random.default_rng([7, seed])
    xn, yn = dx * np.arange(nx + 1), dx * np.arange(ny + 1)
    amp = 1.2 if case["front"] > 0 else 0.4
    z = amp * (1.0 + _smooth(gen, xn, yn, Lx, Ly, 12, 60.0 * dx))
    xc, yc = dx * (np.arange(nx) + 0.5), dx * (np.arange(ny) + 0.5)
    X = torch.as_tensor(xc, device=DEV)[None, :]
    Y = torch.as_tensor(yc, device=DEV)[:, None]
    ripple = _smooth(gen, xc, yc, Lx, Ly, 8, 24.0 * dx)
    depth = float(gen.uniform(2.5, 3.5))
    if case["front"] > 0:
        R = case["front"] * min(Lx, Ly)
        dxr, dyr = X - 0.5 * Lx, Y - 0.5 * Ly
        r = torch.sqrt(dxr * dxr + dyr * dyr) / R
        h = depth * (1.0 - r).clamp(min=0.0) ** 1.5 * (1.0 + 0.1 * ripple)
        speed = 1.5 * math.sqrt(G * depth)
        u, v = speed * dxr / R, speed * dyr / R
    else:
        b = 0.25 * (z[1:, 1:] + z[:-1, 1:] + z[1:, :-1] + z[:-1, :-1])
        step = torch.where(X < 0.5 * Lx, 0.75, 0.0)  # a dam break inside the basin
        h = depth + step + 0.1 * ripple - b
        u, v = 0.3 * ripple, -0.2 * ripple.flip(0)
        speed = 1.0
    h = h.clamp(min=0.0) + torch.zeros_like(X + Y)
    hu, hv = h * u, h * v
    dt0 = 0.5 * cfl * dx / (speed + 1.2 * math.sqrt(G * (depth + 1.0)))
    return cfg, z, h, hu, hv, dt0


def _to_patches(a, mi, mj, m):
    """[ny][nx] -> [patch][m][m] in Morton order of the patches."""
    def key(q):
        x, y = q
        return sum(((x >> i) & 1) << (2 * i) | ((y >> i) & 1) << (2 * i + 1) for i in range(12))
    order = sorted(((x, y) for y in range(mj) for x in range(mi)), key=key)
    t = a.reshape(mj, m, mi, m).permute(0, 2, 1, 3).reshape(mj * mi, m, m)
    return t[torch.as_tensor([y * mi + x for x, y in order], device=a.device)].contiguous()


def _valley_problem(case, seed, scen=0):
    """V-valley of 250 m blocks (side slope 0.05, down-valley slope 0.005,
    noise 0.5 m), reservoir upstream of the breach, DEM nodes every 8 m."""
    gen = np.random.default_rng([11, seed, scen])
    side = 250.0 if case["kind"] == "amr" else 500.0
    Lx, Ly = side * case["mi"], side * case["mj"]
    breach = 0.15 * Lx
    prob = inputs.v_valley(mi=case["mi"], mj=case["mj"], patch=case["mx"],
                           minlevel=case.get("minlevel", 0), maxlevel=case["maxlevel"],
                           seed=int(gen.integers(1 << 30)), dem_spacing=8.0,
                           depth=float(gen.uniform(10.0, 14.0) if case["kind"] == "advance"
                                       else gen.uniform(17.0, 21.0)),
                           breach_x=breach, manning_n=float(gen.uniform(0.025, 0.04)),
                           n_gauges=8, Lx=Lx, Ly=Ly,
                           breach_width=float(gen.uniform(80.0, 300.0))
                           if case.get("nscen", 1) > 1 else None)
    prob.cfg.precision = case["precision"]
    prob.cfg.src_level = case["maxlevel"]
    return prob


def _tongue(prob, reach):
    """Mid-flood state of a valley: the reservoir, then a tongue whose surface
    falls parabolically to the thalweg's bed over `reach` metres, running
    down-valley."""
    cfg = prob.cfg
    x0 = cfg.src_box[1]
    surf0 = cfg.eta0

    def ic(x, y, b):
        xi = np.clip((x - x0) / reach, 0.0, 1.0)
        bed_front = 0.005 * (cfg.xupper - (x0 + reach)) - 0.5
        surf = np.where(x < x0, surf0, bed_front + (surf0 - bed_front) * (1.0 - xi) ** 2)
        h = np.maximum(surf - b, 0.0)
        u = np.where(x < x0, 0.0, 6.0 * xi)
        return h, h * u, 0.05 * h * u * np.sin(y / 40.0)
    return ic


def _refined(f, ic, levels, s=0):
    for _ in range(levels):
        f.set_state(ic, s)
        f.regrid()
    f.set_state(ic, s)


def _read_bufs(cap, m):
    return [_pinned((cap, m, m)) for _ in range(3)]


def prepare(case, seed):
    return {"uniform": _prep_window, "amr": _prep_window, "advance": _prep_advance,
            "inflow": _prep_inflow, "tiles": _prep_tiles, "grad": _prep_grad}[case["kind"]](case, seed)


def _prep_window(case, seed):
    if case["kind"] == "uniform":
        cfg, z, h, hu, hv, dt0 = _uniform_input(case, seed)
        dem = inputs.Dem(z.cpu().numpy(), 0.0, 0.0, case["dx"], case["dx"])
        cap = cfg.mi * cfg.mj
        f = geoflood.Forest(cfg, dem, max_patches=cap)
        q = [_pinned(tuple([cfg.mi * cfg.mj, cfg.mx, cfg.mx])) for _ in range(3)]
        for d, a in zip(q, (h, hu, hv)):
            d.copy_(_to_patches(a, cfg.mi, cfg.mj, cfg.mx))
    else:
        if case["terrain"] == "valley":
            prob = _valley_problem(case, seed)
            ic = _tongue(prob, 0.25 * (prob.cfg.xupper - prob.cfg.src_box[1]))
        else:
            prob = inputs.canyon_plain(patch=case["mx"], minlevel=case["minlevel"],
                                       maxlevel=case["maxlevel"], seed=seed & 0xffff,
                                       dem_spacing=40.0, precision=case["precision"])
            ic = prob.ic
        cap = 26000 if case["terrain"] == "canyon" else 12000
        f = geoflood.Forest(prob.cfg, prob.dem, max_patches=cap)
        _refined(f, ic, case["maxlevel"] - case["minlevel"])
        f.set_gauges(prob.gauges)
        cfg = prob.cfg
        q = [_pinned(a.shape).copy_(torch.from_numpy(a)) for a in f.read()[:3]]
        assert len(q[0]) <= cap
        dt0 = 0.02 * (cfg.xupper - cfg.xlower) / (cfg.mi * cfg.mx << cfg.maxlevel)
    n = len(q[0])
    out = [_pinned((max(cap, n), cfg.mx, cfg.mx)).zero_() for _ in range(3)]
    f32 = [torch.zeros(a.shape, dtype=torch.float32) for a in out] if case["precision"] else None
    return dict(kind="window", f=f, q=[a.numpy() for a in q], out=out, steps=case["steps"],
                dt0=dt0, f32=f32, n=n)


def _advance_state(f, case, cap):
    out = [_pinned((cap, case["mx"], case["mx"])) for _ in range(3)]
    f32 = [torch.empty(a.shape, dtype=torch.float32) for a in out] if case["precision"] else None
    for a in out + (f32 or []):
        a.zero_()
    return dict(kind="advance", f=f, ckpt=f.save(), out=out, f32=f32, t_end=case["t_end"],
                forest=np.full((cap, 3), -1, np.int32),
                regrid=case.get("regrid", 4), check=case.get("check", 4),
                on_miss=bool(case.get("learned", 0)), nscen=case.get("nscen", 1))


def _prep_advance(case, seed):
    n = case["nscen"]
    probs = [_valley_problem(case, seed, s) for s in range(n)]
    cap = max(64, n * case["mi"] * case["mj"] * 4 ** case["maxlevel"])
    f = geoflood.Forest(probs[0].cfg, None, num_scenarios=n, max_patches=cap)
    for s, p in enumerate(probs):
        f.set_scenario(s, p.cfg.manning_n, p.cfg.eta0)
        f.set_topo(p.dem, s)
    for k in range(case["maxlevel"] + 1):
        for s, p in enumerate(probs):
            f.set_state(p.ic, s)
        if k < case["maxlevel"]:
            f.regrid()
    for s, p in enumerate(probs):
        f.set_gauges(p.gauges, s)
        f.set_time(0.0, 0.01, s)
    if case["learned"]:
        f.cnn_set_params(inputs.cnn_init(seed & 0xffff))
        f.set_tagger(geoflood.TAGGER_LEARNED, 0.8)
    return _advance_state(f, case, cap)


def _prep_inflow(case, seed):
    gen = np.random.default_rng([13, seed])
    prob = inputs.flood_speed(patch=case["mx"], maxlevel=case["maxlevel"],
                              precision=case["precision"], peak=case["peak"])
    cfg = prob.cfg
    q = case["peak"] * float(gen.uniform(0.9, 1.1))
    cfg.hydrograph = ((0.0, 0.2 * q), (300.0, q), (14400.0, q), (18000.0, 0.0))
    xn, yn = np.arange(0.0, 1001.0, 20.0), np.arange(0.0, 2001.0, 20.0)
    z = 0.02 * _smooth(gen, xn, yn, 1000.0, 2000.0, 8, 300.0).cpu().numpy()
    f = geoflood.Forest(cfg, inputs.Dem(z, 0.0, 0.0, 20.0, 20.0), max_patches=2 * 4 ** case["maxlevel"])
    _refined(f, prob.ic, case["maxlevel"])
    f.set_time(0.0, cfg.dt_initial)
    return _advance_state(f, case, 2 * 4 ** case["maxlevel"])


def _tile_input(case, seed):
    """q [n][3][T][T], b [n][T][T] with ghosts, dx, dt, manning: swells of
    varying depth over rolling beds, some tiles' corners dry."""
    m, n = case["mx"], case["npatch"]
    T = m + 4
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + n)
    dx = 2.0

    def waves(amp, count=4):
        x = torch.arange(T, dtype=torch.float64, device=DEV)
        out = torch.zeros(n, T, T, dtype=torch.float64, device=DEV)
        for _ in range(count):
            k = torch.rand(n, 3, 1, 1, generator=g, dtype=torch.float64, device=DEV)
            out += torch.sin(0.5 * (k[:, 0] * x[None, None, :] + k[:, 1] * x[None, :, None])
                             + 6.28 * k[:, 2])
        return amp / count * out
    b = 1.0 + waves(1.5)
    eta = 1.0 + waves(0.5) + torch.rand(n, 1, 1, generator=g, dtype=torch.float64, device=DEV)
    wet = torch.rand(n, 1, 1, generator=g, dtype=torch.float64, device=DEV) < case["wet"]
    h = torch.where(wet, (eta - b).clamp(min=0.0), torch.zeros_like(b))
    q = torch.stack([h, h * waves(2.0), h * waves(2.0)], 1).contiguous()
    return q, b.contiguous(), dx, 0.1, 0.03


def _prep_tiles(case, seed):
    q, b, dx, dt, mn = _tile_input(case, seed)
    L = geoflood.lib()
    fn = L.geoflood_step_tiles_noalloc
    vp, d = ctypes.c_void_p, ctypes.c_double
    fn.argtypes = [vp, vp, vp, ctypes.c_int, ctypes.c_int, d, d, d, d, d, d, vp, vp]
    fn.restype = ctypes.c_int
    return dict(kind="tiles", fn=fn, q=q, b=b, out=torch.empty_like(q), n=case["npatch"],
                m=case["mx"], dx=dx, dt=dt, mn=mn, cmax=ctypes.c_double())


def _grad_input(case, seed):
    """BF16 bits of n samples [n][324][16] (five live channels of smooth
    fields, the rest zero), labels, parameters."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 104729 + 17)
    n = case["n"]
    x = torch.zeros(n, 18, 18, 16, device=DEV)
    low = torch.randn(n, 5, 5, 5, generator=g, device=DEV)
    x[..., :5] = torch.nn.functional.interpolate(low, (18, 18), mode="bilinear").permute(0, 2, 3, 1)
    bits = x.reshape(n, 324, 16).to(torch.bfloat16).view(torch.int16)
    y = (torch.rand(n, generator=g, device=DEV) < 0.2).float()
    return bits, y, inputs.cnn_init(seed & 0xffff)


def _prep_grad(case, seed):
    bits, y, prm = _grad_input(case, seed)
    f = geoflood.Forest(inputs.Config(mi=1, mj=1, mx=32))
    f.cnn_set_params(prm)
    return dict(kind="grad", f=f, x=bits.cpu().numpy().view(np.uint16), y=y.cpu().numpy(),
                pw=case["pos_weight"])


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _result(out, f32, n):
    """The caller's buffers, the first n patches just read (the rest of their
    capacity unused); single precision for an FP32 context."""
    if f32 is None:
        return out
    for d, a in zip(f32, out):
        d[:n].copy_(a[:n])
    return f32


def run(state):
    k = state["kind"]
    if k == "window":
        f = state["f"]
        f.write(*state["q"])
        f.set_time(0.0, state["dt0"])
        t, _ = f.step(1e9, state["steps"])
        f.read_into(*[a.numpy() for a in state["out"]])
        return {"q": _result(state["out"], state["f32"], state["n"]), "t": t}
    if k == "advance":
        f, nscen = state["f"], state["nscen"]
        f.load(state["ckpt"])
        f.advance(state["t_end"], state["regrid"], state["check"], regrid_on_miss=state["on_miss"])
        n, forest = 0, state["forest"]
        for s in range(nscen):
            info = f.patch_info(s)
            m = n + info[0].shape[0]
            for a in range(3):
                forest[n:m, a] = info[a]
            f.read_into(*[a[n:m].numpy() for a in state["out"]], s=s)
            n = m
        return {"q": _result(state["out"], state["f32"], n), "forest": forest}
    if k == "tiles":
        st = state
        rc = st["fn"](st["q"].data_ptr(), st["b"].data_ptr(), st["out"].data_ptr(), st["n"], st["m"],
                      st["dx"], st["dx"], st["dt"], G, 1e-3, st["mn"], ctypes.addressof(st["cmax"]),
                      torch.cuda.current_stream().cuda_stream)
        if rc:
            raise RuntimeError("step_tiles_noalloc: %d" % rc)
        return {"q": st["out"], "cmax": st["cmax"].value}
    logit, grad, loss = state["f"].cnn_grad(state["x"], state["y"], state["pw"])
    return {"logit": logit, "grad": grad, "loss": np.float32(loss)}


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: the pass's inputs once, its outputs once, and per step the state
    and bed read and the state written (FP64 56 B, FP32 40 B per cell).  FLOPs:
    468 per wet cell and step of the scheme's own operations."""
    k = case["kind"]
    if k == "grad":
        fl = 3 * (2.0 * 256 * 16 * 144) * 3 * case["n"]
        return {"bytes": case["n"] * (324 * 32 + 8) + 3 * 4 * 6977, "flops": fl}
    if k == "tiles":
        T2 = (case["mx"] + 4) ** 2
        return {"bytes": case["npatch"] * T2 * 8 * 7,
                "flops": 468.0 * case["npatch"] * case["mx"] ** 2 * 0.7 * case["wet"]}
    per = 40 if case["precision"] else 56
    m2 = case["mx"] ** 2
    if k == "uniform":
        cells, steps = case["mi"] * case["mj"] * m2, case["steps"]
        r = min(case["mi"], case["mj"]) * case["mx"] * case["front"]
        wet = min(cells, math.pi * r * r) if case["front"] > 0 else cells
    elif k == "amr":
        # patches: the base grid and the refined reservoir and tongue
        if case["terrain"] == "canyon":
            cells, wet = 19350 * m2, 4.0e5
        else:
            base = case["mi"] * case["mj"] * 4 ** case["maxlevel"]
            cells, wet = 0.32 * base * m2, 0.14 * base * m2
        steps = case["steps"]
    elif k == "advance":
        base = case["nscen"] * case["mi"] * case["mj"] * 4 ** case["maxlevel"]
        cells, wet = 0.23 * base * m2, 0.06 * base * m2
        dx = 500.0 / (case["mx"] * 2 ** case["maxlevel"])
        steps = case["t_end"] * 20.0 / (0.9 * dx)
    else:
        cells, wet = 20 * m2, 2.3 * m2
        dx = 1000.0 / (case["mx"] * 2 ** case["maxlevel"])
        steps = case["t_end"] * 3.8 / (0.9 * dx)
    return {"bytes": cells * (48 + per * steps), "flops": 468.0 * wet * steps}


# ---------------------------------------------------------------------------
# 64-bit values of the outputs, by plain torch
# ---------------------------------------------------------------------------

def _riemann(l, r, g, dry):
    """Augmented solver with f-waves, elementwise.  l, r: (h, n, t, b).
    Returns waves Z[3][3] and speeds s[3]."""
    W, Z0 = torch.where, torch.zeros_like(l[0])
    hl, nl, tl, bl = l
    hr, nr, tr, br = r
    wl, wr = hl > dry, hr > dry
    el, er = hl, hr
    hl, nl, tl = W(wl, hl, Z0), W(wl, nl, Z0), W(wl, tl, Z0)
    hr, nr, tr = W(wr, hr, Z0), W(wr, nr, Z0), W(wr, tr, Z0)
    one = torch.ones_like(hl)
    # a dry side above the other side's surface: wall, or overtopped
    cl, cr = torch.sqrt(g * hl), torch.sqrt(g * hr)
    dryr = wl & ~wr & (br > hl + bl)
    sw = torch.maximum(cl - nl / W(wl, hl, one), cl)
    wallr = dryr & (br >= bl + hl + nl / W(sw > 0, sw, one))
    dryl = wr & ~wl & (bl > hr + br)
    sw = torch.maximum(nr / W(wr, hr, one) + cr, cr)
    walll = dryl & (bl >= br + hr - nr / W(sw > 0, sw, one))
    br = W(dryr & ~wallr, hl + bl, br)
    bl = W(dryl & ~walll, hr + br, bl)
    hr, nr, tr, br, er = (W(wallr, x, y) for x, y in ((hl, hr), (-nl, nr), (tl, tr), (bl, br), (hl, er)))
    hl, nl, tl, bl, el = (W(walll, x, y) for x, y in ((hr, hl), (-nr, nl), (tr, tl), (br, bl), (hr, el)))
    pl, pr = hl > 0, hr > 0
    ul, vl = W(pl, nl / W(pl, hl, one), Z0), W(pl, tl / W(pl, hl, one), Z0)
    ur, vr = W(pr, nr / W(pr, hr, one), Z0), W(pr, tr / W(pr, hr, one), Z0)
    cl, cr = torch.sqrt(g * hl), torch.sqrt(g * hr)
    ql, qr = torch.sqrt(hl), torch.sqrt(hr)
    uh = (ql * ul + qr * ur) / W(pl | pr, ql + qr, one)
    ch = torch.sqrt(g * (0.5 * (hl + hr)))
    s1 = W(pl & pr, torch.minimum(ul - cl, uh - ch), W(pr, ur - 2 * cr, ul - cl))
    s3 = W(pl & pr, torch.maximum(ur + cr, uh + ch), W(pr, ur + cr, ul + 2 * cl))
    s2 = 0.5 * (s1 + s3)
    any_ = pl | pr
    den = W(any_, s3 - s1, one)
    db, dn = br - bl, nr - nl
    deta = (er + br) - (el + bl)
    hh = (s3 * hr - s1 * hl - dn) / den
    sub, right = (s1 < 0) & (s3 > 0), s1 >= 0
    q1, q3 = hh * den / W(s1 != 0, s1, one), hh * den / W(s3 != 0, s3, one)
    lo = W(sub, q1, W(right, -hl, W(s3 < 0, q3, -db)))
    hi = W(sub, q3, W(right, W(s1 > 0, q1, -db), hr))
    d = -db
    below = d < lo
    dc = W(below, lo, d)
    above = dc > hi
    dc = W(above, hi, dc)
    # transcritical left-going: bounds apply in the order lo, hi; right-going: hi, lo
    dr = W(d > hi, hi, d)
    dr = W(dr < lo, lo, dr)
    dhs = W(right, dr, dc)
    d1 = W(dhs != d, (hr - hl) - dhs, deta)
    d3 = (nr * ur - nl * ul) + g * (0.5 * (hl + hr)) * deta
    b1, b3 = (s3 * d1 - dn) / den, (dn - s1 * d1) / den
    b2 = d3 - (s1 * s1 * b1 + s3 * s3 * b3)
    Z = [[s1 * b1, s1 * s1 * b1, vl * s1 * b1], [Z0, b2, Z0], [s3 * b3, s3 * s3 * b3, vr * s3 * b3]]
    Z[1][2] = (nr * vr - nl * vl) - (Z[0][2] + Z[2][2])
    for p in range(3):
        off = ~any_ | (wallr & (p > 0)) | (walll & (p < 2))
        Z[p] = [W(off, Z0, z) for z in Z[p]]
    return Z, [W(any_, s, Z0) for s in (s1, s2, s3)]


def _sweep(q, b, nu, nut, g, dry):
    """x sweep of tiles q (h, n, t) [..., Y, X] with two ghost cells.  Returns
    nu dQ of the interior cells, the transverse fluxes on the y edges
    [..., M+1, M] (h, n, t) and the largest speed."""
    W = torch.where
    h = q[0]
    L = [a[..., 1:-1, :-1] for a in (*q, b)]
    R = [a[..., 1:-1, 1:] for a in (*q, b)]
    Z, s = _riemann(L, R, g, dry)
    zero = torch.zeros_like(s[0][..., 1:-1])
    am, ap, ff = [zero] * 3, [zero] * 3, [zero] * 3
    wet = (h > dry)[..., 1:-1, :]
    both = wet[..., 1:-2] & wet[..., 2:-1]
    smax = 0.0
    for p in range(3):
        sp = s[p][..., 1:-1]
        smax = max(smax, float(sp[..., 1:-1, :].abs().max()))
        z = [a[..., 1:-1] for a in Z[p]]
        up = [W(sp > 0, a[..., :-2], a[..., 2:]) for a in Z[p]]
        zz = z[0] ** 2 + z[1] ** 2 + z[2] ** 2
        th = (up[0] * z[0] + up[1] * z[1] + up[2] * z[2]) / W(zz != 0, zz, torch.ones_like(zz))
        phi = torch.minimum(torch.minimum(0.5 * (1 + th), torch.full_like(th, 2.0)), 2 * th).clamp(min=0)
        coef = W(both & (zz != 0), 0.5 * torch.sign(sp) * (1 - nu * sp.abs()) * phi, zero)
        wm = W(sp < 0, 1.0, W(sp == 0, 0.5, 0.0))
        for k in range(3):
            am[k] = am[k] + wm * z[k]
            ap[k] = ap[k] + (1 - wm) * z[k]
            ff[k] = ff[k] + coef * z[k]
    d = [ap[k][..., :-1] + am[k][..., 1:] + (ff[k][..., 1:] - ff[k][..., :-1]) for k in range(3)]
    # transverse split of the increments of lines -1..M along y
    c = (Ellipsis, slice(1, -1), slice(2, -2))
    hc, nc, tc, bc = h[c], q[1][c], q[2][c], b[c]
    wc = hc > dry
    hs = W(wc, hc, torch.ones_like(hc))
    w, z, cc = tc / hs, nc / hs, torch.sqrt(g * hs)
    a1 = ((w + cc) * d[0] - d[2]) / (2 * cc)
    a3 = (d[2] - (w - cc) * d[0]) / (2 * cc)
    a2 = d[1] - z * d[0]
    parts = [(w - cc, (a1, z * a1, (w - cc) * a1)), (w + cc, (a3, z * a3, (w + cc) * a3)),
             (w, (torch.zeros_like(a2), a2, torch.zeros_like(a2)))]
    eta = hc + bc
    hy, by = h[..., 2:-2], b[..., 2:-2]
    openp = ~(~(hy[..., 2:, :] > dry) & (by[..., 2:, :] > eta)) & wc
    openm = ~(~(hy[..., :-2, :] > dry) & (by[..., :-2, :] > eta)) & wc
    tr = []
    for k in range(3):
        plus = sum(W(lam > 0, lam * a[k], torch.zeros_like(lam)) for lam, a in parts)
        minus = sum(W(lam < 0, lam * a[k], torch.zeros_like(lam)) for lam, a in parts)
        plus, minus = W(openp, plus, 0.0), W(openm, minus, 0.0)
        tr.append(-0.5 * nu * (plus[..., :-1, :] + minus[..., 1:, :]))
    return [nu * a[..., 1:-1, :] for a in d], tr, smax


def _step64(q, b, dx, dt, g, dry, mn):
    """One default-scheme step of tiles with filled ghosts; new interior, cmax."""
    nu = dt / dx
    T = lambda a: a.transpose(-1, -2)
    X, Gy, sx = _sweep(q, b, nu, nu, g, dry)
    Yt, Ft, sy = _sweep([T(q[0]), T(q[2]), T(q[1])], T(b), nu, nu, g, dry)
    Y, F = [T(Yt[0]), T(Yt[2]), T(Yt[1])], [T(Ft[0]), T(Ft[2]), T(Ft[1])]
    o = []
    for k in range(3):
        tf = nu * (F[k][..., 1:] - F[k][..., :-1]) + nu * (Gy[k][..., 1:, :] - Gy[k][..., :-1, :])
        o.append(q[k][..., 2:-2, 2:-2] - (X[k] + Y[k]) - tf)
    o[0] = o[0].clamp(min=0.0)
    wet = o[0] > dry
    if mn > 0:
        hs = torch.where(wet, o[0], torch.ones_like(o[0]))
        sp = torch.sqrt((o[1] / hs) ** 2 + (o[2] / hs) ** 2)
        den = 1.0 + dt * g * mn * mn * sp / hs ** (4.0 / 3.0)
        o[1], o[2] = o[1] / den, o[2] / den
    return [o[0]] + [torch.where(wet, a, torch.zeros_like(a)) for a in o[1:]], max(sx, sy) / dx


def _mirror(q):
    """Interior -> two ghost layers of wall mirrors on every side."""
    out = []
    for k, a in enumerate(q):
        sx, sy = (-1.0 if k == 1 else 1.0), (-1.0 if k == 2 else 1.0)
        a = torch.cat([sx * a[..., [1, 0]], a, sx * a[..., [-1, -2]]], -1)
        out.append(torch.cat([sy * a[..., [1, 0], :], a, sy * a[..., [-1, -2], :]], -2))
    return out


def exact(case, seed):
    k = case["kind"]
    if k == "tiles":
        q, b, dx, dt, mn = _tile_input(case, seed)
        o, cm = _step64([q[:, 0], q[:, 1], q[:, 2]], b, dx, dt, G, 1e-3, mn)
        return {"q": torch.stack(_mirror(o), 1), "cmax": cm}
    if k == "grad":
        return _exact_grad(case, seed)
    if k != "uniform" or case["first_order"] or case["no_transverse"] or case["dim_split"]:
        return None
    if case["mi"] * case["mj"] * case["mx"] ** 2 * case["steps"] > 1.2e8:
        return None
    cfg, z, h, hu, hv, dt = _uniform_input(case, seed)
    b = _mirror([0.25 * (z[1:, 1:] + z[:-1, 1:] + z[1:, :-1] + z[:-1, :-1])])[0]
    q, t, n = [h, hu, hv], 0.0, 0
    while n < case["steps"]:
        o, cm = _step64(_mirror(q), b, case["dx"], dt, G, case["drytol"], case["manning"])
        if dt * cm > cfg.cfl_max:
            dt = cfg.cfl_desired / cm
            continue
        q, t, n, dt = o, t + dt, n + 1, cfg.cfl_desired / cm if cm > 0 else dt
    return {"q": [_to_patches(a, cfg.mi, cfg.mj, cfg.mx) for a in q], "t": t}


def _exact_grad(case, seed):
    bits, y, prm = _grad_input(case, seed)
    x = bits.view(torch.bfloat16).double().reshape(-1, 18, 18, 16).permute(0, 3, 1, 2)
    y = y.double()
    p = torch.as_tensor(prm, dtype=torch.float64, device=DEV).requires_grad_(True)
    at = 0
    a = x
    for layer in range(3):
        w = p[at:at + 2304].reshape(16, 3, 3, 16).permute(0, 3, 1, 2)
        bias = p[at + 2304:at + 2320]
        at += 2320
        a = torch.relu(torch.nn.functional.conv2d(a, w, bias, padding=0 if layer == 0 else 1))
    logit = a.mean((2, 3)) @ p[at:at + 16] + p[at + 16]
    wgt = torch.where(y > 0.5, case["pos_weight"], 1.0)
    loss = (wgt * torch.nn.functional.binary_cross_entropy_with_logits(logit, y, reduction="none")).mean()
    loss.backward()
    return {"logit": logit.detach(), "grad": p.grad, "loss": loss.detach()}
