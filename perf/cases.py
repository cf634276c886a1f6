"""Performance cases of the shallow-water library, through its public entry points.

Four kinds of work:

* ``grid``: a context of one uniform grid (``Tsunami.step``), split or unsplit
  scheme, plane or latitude-longitude coordinates, with or without Manning
  friction, in either precision;
* ``block``: one step of a grid in the caller's own device memory
  (``tsu_grid_step_noalloc``);
* ``amr`` and ``ensemble``: a whole run of a refined hierarchy, from the
  creation of the context to the surface on the host;
* ``logits`` and ``grad``: the refinement-flag predictor, inference and the
  gradient of its loss.

Seas: ``uplift`` (still water and the seafloor uplift of the shelf workloads,
the first minutes after an earthquake), ``swell`` (waves and currents
everywhere, a run that has been going for hours) and ``hump`` (the Gaussian
surface hump of the closed basin).

FP32 runs return single-precision arrays and FP64 runs double-precision ones.
"""
import math

import numpy as np
import torch

from paper_1901_06798_gb300 import binding as tsu
from paper_1901_06798_gb300 import workloads as W

G = 9.81
DRYTOL = 1e-3
CFL = 0.9


def listed():
    return [
        # the smallest call: one step of a tiny grid, handed to the library for each step
        dict(name="block_small_f32", kind="block", prec="f32", nx=48, ny=40),
        # the closed basin of the small configuration: a step every few tens of microseconds
        dict(name="pond_f32", kind="grid", prec="f32", bed="pond", sea="hump", nx=200, ny=200, steps=20,
             scheme="split", lonlat=False, manning=0.0),
        # the uniform headline run: 4096 x 4096 cells of 500 m over the shelf
        dict(name="shelf_f32", kind="grid", prec="f32", bed="shelf", sea="uplift", nx=4096, ny=4096, steps=2,
             scheme="split", lonlat=False, manning=0.0),
        # an ocean run as the paper's: degrees, Manning friction, waves everywhere, odd sizes
        dict(name="ocean_f32", kind="grid", prec="f32", bed="shelf", sea="swell", nx=1531, ny=1213, steps=4,
             scheme="split", lonlat=True, manning=0.025),
        # the scheme of the original CPU code (transverse corrections)
        dict(name="unsplit_f32", kind="grid", prec="f32", bed="shelf", sea="swell", nx=1024, ny=1024, steps=4,
             scheme="unsplit", lonlat=False, manning=0.0),
        # a double-precision reference run of a window of the shelf
        dict(name="shelf_f64", kind="grid", prec="f64", bed="shelf", sea="uplift", nx=512, ny=512, steps=4,
             scheme="split", lonlat=False, manning=0.0),
        # steps of grids that another program owns, waves everywhere
        dict(name="block_f32", kind="block", prec="f32", nx=2050, ny=1537),
        dict(name="block_f64", kind="block", prec="f64", nx=771, ny=602),
        # three-level run over the shelf, full size: 2 km down to 125 m
        dict(name="amr_f32", kind="amr", prec="f32", n=1000, steps=16),
        # many earthquakes over one shelf, two levels each
        dict(name="ensemble_f32", kind="ensemble", prec="f32", n=512, scenarios=16, steps=32),
        # the flag predictor: inference on a regrid's window, a training batch's gradient
        dict(name="cnn_logits", kind="logits", n=1, h=700, w=900),
        dict(name="cnn_grad", kind="grad", n=4, h=128, w=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid", "grid64", "block", "block64", "amr", "ensemble", "logits", "grad"])
    if kind in ("grid", "grid64"):
        f64 = kind == "grid64"
        hi = 600 if f64 else 2900
        bed = rng.choice(["pond", "shelf", "shelf"])
        scheme = rng.choice(["split", "split", "unsplit"])
        lonlat = bed == "shelf" and scheme == "split" and rng.random() < 0.4
        return dict(kind="grid", prec="f64" if f64 else "f32", bed=bed,
                    sea="hump" if bed == "pond" else rng.choice(["uplift", "swell"]), nx=_log_int(rng, 64, hi),
                    ny=_log_int(rng, 64, hi), steps=2 * rng.randint(1, 4), scheme=scheme, lonlat=lonlat,
                    manning=rng.choice([0.0, 0.025]))
    if kind in ("block", "block64"):
        f64 = kind == "block64"
        return dict(kind="block", prec="f64" if f64 else "f32", nx=_log_int(rng, 40, 1000 if f64 else 3500),
                    ny=_log_int(rng, 40, 1000 if f64 else 3500))
    if kind == "amr":
        return dict(kind="amr", prec="f32", n=_log_int(rng, 120, 800), steps=4 * rng.randint(2, 4))
    if kind == "ensemble":
        return dict(kind="ensemble", prec="f32", n=_log_int(rng, 128, 512), scenarios=rng.randint(2, 16),
                    steps=4 * rng.randint(4, 8))
    if kind == "logits":
        return dict(kind="logits", n=rng.randint(1, 4), h=_log_int(rng, 48, 700), w=_log_int(rng, 48, 900))
    return dict(kind="grad", n=rng.randint(1, 4), h=_log_int(rng, 32, 160), w=_log_int(rng, 32, 160))


# ------------------------------------------------------------------ inputs


def _swell(gen, Lx, Ly, nodes, total, shortest):
    """Waves in all directions on a (nodes, nodes) node grid over Lx x Ly:
    wavelengths between `shortest` and half the domain, rms height `total`."""
    x = np.linspace(0.0, Lx, nodes)[None, :]
    y = np.linspace(0.0, Ly, nodes)[:, None]
    v = np.zeros((nodes, nodes))
    n = 16
    for lam in np.exp(gen.uniform(np.log(shortest), np.log(max(2.0 * shortest, 0.5 * min(Lx, Ly))), n)):
        a, p = gen.uniform(0.0, 2.0 * np.pi, 2)
        k = 2.0 * np.pi / lam
        v += np.cos(k * (x * np.cos(a) + y * np.sin(a)) + p)
    return v * (total / np.sqrt(0.5 * n))


def _grid_workload(case, seed):
    """The workload (configuration and host input grids) of a `grid` case."""
    gen = np.random.Generator(np.random.PCG64([seed, 1]))
    nx, ny = case["nx"], case["ny"]
    if case["bed"] == "pond":
        dx = 10.0
        Lx, Ly = nx * dx, ny * dx
        cfg = W.base_config(nx=nx, ny=ny, dx=dx, dy=dx, bc=[W.BC_WALL] * 4, cfl_desired=CFL)
        r = 0.075 * min(Lx, Ly)
        eta = W.gaussian_grid(0.0, 0.0, Lx, Ly, 201, 201, Lx * gen.uniform(0.3, 0.7), Ly * gen.uniform(0.3, 0.7),
                              gen.uniform(0.3, 0.7), r, r)
        w = dict(cfg=cfg, topo=W.flat_topo(cfg, 10.0), eta=[(0, *eta)], uplift=[], gauges=np.zeros((0, 2)))
    else:
        dx = 500.0
        Lx, Ly = nx * dx, ny * dx
        scale = Lx / 2048e3
        cfg = W.base_config(nx=nx, ny=ny, dx=dx, dy=dx, bc=[W.BC_EXTRAP] * 4, cfl_desired=CFL)
        w = dict(cfg=cfg, topo=W.shelf_topo(Lx, Ly, scale=scale, step_km=0.5), eta=[], uplift=[],
                 gauges=np.array([[Lx * 0.7, Ly * 0.5], [Lx * 0.85, Ly * 0.5]]))
        if case["sea"] == "uplift":
            up = W.shelf_uplift(Lx, Ly, scale=scale, amp=gen.uniform(1.0, 3.0), s_km=gen.uniform(560.0, 700.0),
                                yc=Ly * gen.uniform(0.4, 0.6))
            w["uplift"] = [(0, *up)]
        else:
            m = 257
            eta, u, v = (_swell(gen, Lx, Ly, m, a, 16 * dx) for a in (0.3, 0.01, 0.01))
            w["eta"] = [(0, eta, 0.0, 0.0, Lx / (m - 1), Ly / (m - 1))]
            w["uv"] = [(0, u, v, 0.0, 0.0, Lx / (m - 1), Ly / (m - 1))]
    cfg["transverse"] = 1 if case["scheme"] == "unsplit" else 0
    cfg["manning_n"] = case["manning"]
    return W.lonlat(w, 140.0, 30.0) if case["lonlat"] else w


BLOCK_DX = 500.0


def _block_state(case, seed):
    """(q0, hu, hv, B) of a `block` case: waves over a sloping ocean floor with a beach, on the GPU."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    nx, ny = case["nx"], case["ny"]
    dt = torch.float64 if case["prec"] == "f64" else torch.float32
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :] / nx
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None] / ny
    r = torch.rand(3, 12, 4, generator=gen, device="cuda", dtype=torch.float64)

    def waves(k, amp):
        v = torch.zeros(ny, nx, device="cuda", dtype=torch.float64)
        for q in range(12):
            a, b, p, s = r[k, q]
            f = 1.0 + 15.0 * s
            v += torch.cos(2.0 * math.pi * (f * (x * torch.cos(6.3 * a) + y * torch.sin(6.3 * a)) + p)) * (0.5 + b)
        return v * (amp / 3.0)

    B = (-3000.0 + 3040.0 * x ** 3 + 30.0 * waves(0, 1.0)).to(dt)
    eta = waves(1, 0.4).to(dt)
    h = torch.clamp(eta - B, min=0.0)
    wet = h >= DRYTOL
    u = waves(2, 0.02).to(dt)
    hu = torch.where(wet, h * u, torch.zeros_like(h))
    hv = torch.where(wet, -0.5 * h * u.flip(0), torch.zeros_like(h))
    return (torch.where(h > 0, eta, B) if case["prec"] == "f32" else h), hu, hv, B


def _block_dt():
    return 0.7 * BLOCK_DX / math.sqrt(G * 3200.0)


def _refined_workload(case, seed):
    gen = np.random.Generator(np.random.PCG64([seed, 2]))
    if case["kind"] == "ensemble":
        return W.ensemble(n_scen=case["scenarios"], n=case["n"], dx=2048e3 / case["n"], seed=int(gen.integers(1 << 30)))
    L = case["n"] * 2000.0
    w = W.amr3(L=L, dx1=2000.0)
    up = W.shelf_uplift(L, L, scale=L / 2000e3, amp=gen.uniform(1.5, 2.5), s_km=gen.uniform(580.0, 640.0),
                        yc=L * gen.uniform(0.45, 0.55))
    w["uplift"] = [(0, *up)]
    return w


def _cnn_inputs(case, seed):
    """Weights, features (eta, depth, |hu|, |hv|, flag planes as a regrid makes them), targets and mask."""
    gen = np.random.Generator(np.random.PCG64([seed, 3]))
    n, h, w = case["n"], case["h"], case["w"]
    y, x = np.mgrid[0:h, 0:w].astype(np.float32) / 64.0
    f = np.zeros((n, 5, h, w), np.float32)
    for k in range(n):
        ph = gen.uniform(0, 6.28, 6).astype(np.float32)
        wave = np.sin(2.1 * x + ph[0]) * np.cos(1.7 * y + ph[1]) + 0.5 * np.sin(5.3 * (x - y) + ph[2])
        f[k, 0] = 1.5 * wave
        f[k, 1] = np.clip(2.0 + 2.0 * np.sin(0.7 * x + ph[3]), -1, 5)
        f[k, 2] = np.abs(3.0 * np.cos(2.3 * x + ph[4]))
        f[k, 3] = np.abs(2.0 * np.cos(1.9 * y + ph[5]))
        f[k, 4] = (np.abs(wave) > 0.8).astype(np.float32)
    target = np.maximum(f[:, 4], np.roll(f[:, 4], 2, axis=2))
    mask = np.ones((n, h, w), np.float32)
    mask[:, : h // 8] = 0.0
    theta = W.cnn_init_params(int(gen.integers(1 << 30))).astype(np.float32)
    theta[gen.integers(0, theta.size, 64)] += np.float32(0.05)
    return theta, f, target, mask


# ------------------------------------------------------------------ one pass


class _Device:
    """A strided device array of the library's, as the CUDA array interface
    describes it; a tensor over it keeps this object, and so the context, alive."""

    def __init__(self, owner, ptr, shape, strides, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = dict(data=(ptr, False), shape=shape, strides=strides, typestr=typestr, version=3)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "grid":
        w = _grid_workload(case, seed)
        ctx = W.load(tsu.Tsunami(w["cfg"], precision=tsu.TSU_F64 if case["prec"] == "f64" else tsu.TSU_F32P), w)
        ptrs, pitch = ctx.level1_buffers()   # current again after an even number of steps
        b = 8 if case["prec"] == "f64" else 4
        out = [torch.as_tensor(_Device(ctx, p + (2 * pitch + 2) * b, (case["ny"], case["nx"]), (pitch * b, b), "<f%d" % b),
                               device="cuda") for p in ptrs[:3]]
        return dict(kind=kind, ctx=ctx, steps=case["steps"], out=out)
    if kind == "block":
        q = _block_state(case, seed)
        ny, nx = q[0].shape
        pitch = (nx + 4 + 3) // 4 * 4
        block = torch.zeros(7, ny + 4, pitch, device="cuda", dtype=q[0].dtype)
        for f, a in zip((0, 1, 2, 6), q):
            block[f, 2:ny + 2, 2:nx + 2] = a
        args = (tsu.TSU_F64 if case["prec"] == "f64" else tsu.TSU_F32P, block.data_ptr(), nx, ny, pitch,
                pitch * (ny + 4), 0, BLOCK_DX, BLOCK_DX, _block_dt(), G, DRYTOL, [W.BC_EXTRAP] * 2 + [W.BC_WALL] * 2,
                torch.cuda.current_stream().cuda_stream)
        return dict(kind=kind, block=block, args=args, out=[block[f, 2:ny + 2, 2:nx + 2] for f in (3, 4, 5)])
    if kind in ("amr", "ensemble"):
        return dict(kind=kind, w=_refined_workload(case, seed), steps=case["steps"])
    return dict(kind=kind, x=_cnn_inputs(case, seed))


def run(state):
    kind = state["kind"]
    if kind == "grid":
        t = state["ctx"].step(state["steps"], allow_cfl=True)
        return dict(t=float(t[0]), q=state["out"])
    if kind == "block":
        rc, speeds = tsu.tsu_grid_step_noalloc(*state["args"])
        if rc != tsu.TSU_OK:
            raise RuntimeError("tsu_grid_step_noalloc: %d" % rc)
        return dict(speeds=list(speeds), q=state["out"])
    if kind in ("amr", "ensemble"):
        cfg = state["w"]["cfg"]
        ctx = W.load(tsu.Tsunami(cfg, precision=tsu.TSU_F32P), state["w"])
        t = ctx.step(state["steps"], allow_cfl=True)
        n, dx = cfg["nx"], cfg["dx"]
        raster = (n, n, 0.5 * dx, 0.5 * dx, dx, dx)
        maps = [ctx.read_field(s, 0, "eta", *raster).astype(np.float32) for s in range(cfg["n_scenarios"])]
        if kind == "amr":
            maps += [ctx.read_field(0, 0, f, *raster).astype(np.float32) for f in ("hu", "hv")]
        records = ctx.read_gauges(state["steps"])[1].astype(np.float32)
        ctx.close()
        return dict(t=t.astype(np.float32), maps=maps, gauges=records)
    theta, x, target, mask = state["x"]
    if kind == "logits":
        return tsu.cnn_forward(theta, x, fp16=True)
    loss, grad = tsu.cnn_loss_grad(theta, x, target, mask)
    return dict(loss=float(loss), grad=grad)


# ------------------------------------------------------------------ work of one pass

FLOPS = 365.5   # of one cell update of the split scheme, counted in the reference arithmetic


def work(case):
    kind = case["kind"]
    if kind in ("grid", "block"):
        cells = case["nx"] * case["ny"] * case.get("steps", 1)
        unsplit = case.get("scheme") == "unsplit"
        return dict(bytes=cells * (56 if case["prec"] == "f64" else 28), flops=cells * FLOPS * (1.6 if unsplit else 1.0))
    if kind == "amr":
        # level 1, and the shelf strip, the uplift and their buffers (about a tenth of the domain) on
        # levels 2 and 3, which take 4 and 16 steps for each of level 1's
        cells = case["steps"] * case["n"] ** 2 * (1.0 + 0.1 * (4 * 16 + 16 * 256))
        return dict(bytes=cells * 28, flops=cells * FLOPS)
    if kind == "ensemble":
        cells = case["steps"] * case["scenarios"] * case["n"] ** 2 * (1.0 + 0.02 * 4 * 16)
        return dict(bytes=cells * 28, flops=cells * FLOPS)
    px = case["n"] * case["h"] * case["w"]
    macs = 9 * (5 * 16 + 16 * 16 + 16 * 16) + 16
    if kind == "logits":
        return dict(bytes=px * 24, flops=2 * macs * px)
    return dict(bytes=px * 28, flops=2 * px * (3 * macs - 9 * 5 * 16))


# ------------------------------------------------------------------ the same in 64 bits
# One uniform grid in plain torch, depth and momenta in 64 bits.  Cells are
# (h, normal momentum, transverse momentum, B) with two ghost cells per side;
# every function works along the last axis.


def _cell(h, hn, ht, B):
    wet = h >= DRYTOL
    hs = torch.where(wet, h, torch.ones_like(h))
    z = torch.zeros_like(h)
    c = torch.where(wet, torch.sqrt(G * hs), z)
    return dict(h=h, hn=hn, ht=ht, B=B, wet=wet, u=torch.where(wet, hn / hs, z), v=torch.where(wet, ht / hs, z), c=c,
                s=torch.where(wet, torch.sqrt(hs), z))


def _at(z, a, b):
    return {k: v[..., a:b] for k, v in z.items()}


def _pick(m, a, b):
    return {k: torch.where(m, a[k], b[k]) for k in a}


def _mirror(z):
    return dict(z, hn=-z["hn"], u=-z["u"])


def _waves(z):
    """f-waves (3 x 3), speeds (3) and walls of the edges between neighbouring cells."""
    n = z["h"].shape[-1]
    L, R = _at(z, 0, n - 1), _at(z, 1, n)
    lw, rw = L["wet"], R["wet"]
    dead = ~lw & ~rw

    def reach(a, other):   # the surface that water running at a dry cell comes up to stays under its bed
        a_ = torch.clamp(a, min=0.0)
        return a_ * a_ / G + other

    wall_r = lw & ~rw & (reach(L["c"] + 0.5 * L["u"], L["B"]) <= R["B"])
    wall_l = ~lw & rw & (reach(R["c"] - 0.5 * R["u"], R["B"]) <= L["B"])
    L, R = _pick(wall_l, _mirror(R), L), _pick(wall_r, _mirror(L), R)
    lw, rw = L["wet"], R["wet"]
    both = lw & rw
    one = torch.ones_like(L["h"])
    uh = (L["s"] * L["u"] + R["s"] * R["u"]) / torch.where(both, L["s"] + R["s"], one)
    ch = torch.sqrt(G * 0.5 * (L["h"] + R["h"]).clamp(min=0.0))
    s1 = torch.where(both, torch.minimum(L["u"] - L["c"], uh - ch),
                     torch.where(lw, L["u"] - L["c"], R["u"] - 2.0 * R["c"]))
    s3 = torch.where(both, torch.maximum(R["u"] + R["c"], uh + ch),
                     torch.where(lw, L["u"] + 2.0 * L["c"], R["u"] + R["c"]))
    s2 = torch.where(both, uh, torch.where(lw, L["u"], R["u"]))
    deta = (R["h"] + R["B"]) - (L["h"] + L["B"])
    d2 = R["hn"] - L["hn"]
    d3 = (R["hn"] * R["u"] - L["hn"] * L["u"]) + G * 0.5 * (L["h"] + R["h"]) * deta
    d4 = R["hn"] * R["v"] - L["hn"] * L["v"]
    den = torch.where(dead, one, s3 - s1)
    # the depth jump at the bed step, moved where a state of the fan would be negative
    M = s3 * R["h"] - s1 * L["h"] - d2
    delta = L["B"] - R["B"]
    s1n, s3n = torch.where(s1 == 0, one, s1), torch.where(s3 == 0, one, s3)
    sub, sup = (s1 < 0) & (s3 > 0), s1 >= 0
    a = sub & (M - s3 * delta < 0)
    b = sub & ~a & (M - s1 * delta < 0)
    c = sup & (L["h"] + delta < 0)
    d = sup & ~c & (s1 > 0) & (M - s1 * delta < 0)
    rest = ~sub & ~sup
    e = rest & (R["h"] - delta < 0)
    f = rest & ~e & (s3 < 0) & (M - s3 * delta < 0)
    moved = a | b | c | d | e | f
    delta = torch.where(a | f, M / s3n, torch.where(b | d, M / s1n, torch.where(c, -L["h"], torch.where(e, R["h"], delta))))
    d1 = torch.where(moved, (R["h"] - L["h"]) - delta, deta)
    w1m, w1n = (s3 * d1 - d2) / den, (s3 * d2 - d3) / den
    Z0 = [s1 * w1m, s1 * w1n, s1 * w1m * L["v"]]
    Z2 = [s3 * (d1 - w1m), s3 * (d2 - w1n), s3 * (d1 - w1m) * R["v"]]
    nil = torch.zeros_like(one)
    Z = [Z0, [nil, nil, d4 - Z0[2] - Z2[2]], Z2]
    Z = [[torch.where(dead, nil, q) for q in p] for p in Z]
    return Z, [torch.where(dead, nil, s) for s in (s1, s2, s3)], wall_l, wall_r


def _limited(z, r):
    """A-dQ, A+dQ and F~ of the inner edges (all but the first and last), and their largest |speed|; r = dt / dx."""
    Z, s, wl, wr = _waves(z)
    i = slice(1, -1)
    am, ap, F = [0.0] * 3, [0.0] * 3, [0.0] * 3
    for p in range(3):
        sp = s[p][..., i]
        Zi = [q[..., i] for q in Z[p]]
        ZI = [torch.where(sp >= 0, q[..., :-2], q[..., 2:]) for q in Z[p]]
        nn = Zi[0] ** 2 + Zi[1] ** 2 + Zi[2] ** 2
        th = (ZI[0] * Zi[0] + ZI[1] * Zi[1] + ZI[2] * Zi[2]) / torch.where(nn == 0, torch.ones_like(nn), nn)
        phi = torch.clamp(torch.minimum(0.5 * (1.0 + th), torch.clamp(2.0 * th, max=2.0)), min=0.0)
        phi = torch.where(nn == 0, torch.zeros_like(phi), phi)
        cf = 0.5 * torch.sign(sp) * (1.0 - r * sp.abs()) * phi
        left = torch.where(sp < 0, 1.0, torch.where(sp == 0, 0.5, 0.0))
        for m in range(3):
            am[m], ap[m], F[m] = am[m] + left * Zi[m], ap[m] + (1.0 - left) * Zi[m], F[m] + cf * Zi[m]
    wl, wr = wl[..., i], wr[..., i]
    nil = torch.zeros_like(am[0])
    for m in range(3):
        am[m], ap[m] = torch.where(wl, nil, am[m]), torch.where(wr, nil, ap[m])
        F[m] = torch.where(wl | wr, nil, F[m])
    return am, ap, F, torch.maximum(-s[0][..., i], s[2][..., i])


def _post(h, hu, hv):
    h = torch.clamp(h, min=0.0)
    dry = h < DRYTOL
    return h, hu.masked_fill(dry, 0.0), hv.masked_fill(dry, 0.0)


def _drag(h, hu, hv, n, dt):
    if not n:
        return h, hu, hv
    wet = h >= DRYTOL
    D = n * n * G * torch.where(wet, h, torch.ones_like(h)) ** (-7.0 / 3.0) * torch.sqrt(hu * hu + hv * hv)
    f = torch.where(wet, 1.0 + dt * D, torch.ones_like(D))
    return h, hu / f, hv / f


def _T(*a):
    return [x.transpose(-1, -2) for x in a]


def _sphere(g):
    """Capacities of the rows (ghost rows included) and lengths of their lower edges; ones on a plane grid."""
    rows = np.arange(-2, g["ny"] + 2)
    if not g["lonlat"]:
        k = np.ones(rows.size)
        return torch.from_numpy(k).cuda(), torch.from_numpy(np.ones(rows.size + 1)).cuda()
    d = math.pi / 180.0
    lat = lambda j: (g["y0"] + j * g["ddy"]) * d  # noqa: E731
    k = (np.sin(lat(rows + 1)) - np.sin(lat(rows))) / (g["ddy"] * d)
    return torch.from_numpy(k).cuda(), torch.from_numpy(np.cos(lat(np.arange(-2, g["ny"] + 3)))).cuda()


def _split(q, B, g, dt):
    """One split step of the ghost-filled state q; returns the interior and the largest x and y speeds."""
    h, hu, hv = q
    kap, ced = _sphere(g)
    am, ap, F, sx = _limited(_cell(h, hu, hv, B), (dt / g["dx"] / kap)[:, None])
    rx = (dt / g["dx"] / kap)[:, None]
    new = [x[:, 2:-2] - rx * (ap[m][:, :-1] + am[m][:, 1:] + F[m][:, 1:] - F[m][:, :-1]) for m, x in enumerate(q)]
    h, hu, hv = _post(*new)
    smx = float((sx[2:-2] / kap[2:-2, None]).max())
    kb = 0.5 * (kap[1:-2] + kap[2:-1])   # edges 0 .. ny
    ce = ced[2:-2]
    z = _cell(*_T(h, hv, hu, B[:, 2:-2]))
    am, ap, F, sy = _limited(z, (dt * ce / (kb * g["dy"]))[None, :])
    smy = float((sy * (ce / kb)[None, :]).max())
    up = [ce * (ap[m] - F[m]) for m in range(3)], [ce * (am[m] + F[m]) for m in range(3)]
    tot = [up[0][m][:, :-1] + up[1][m][:, 1:] for m in range(3)]
    hvi = hv[2:-2].transpose(0, 1)
    tot[0] = tot[0] + (ce[1:] - ce[:-1]) * hvi
    ry = dt / (kap[2:-2] * g["dy"])
    n0, n1, n2 = (a[:, 2:-2] - ry * t for a, t in zip(_T(h, hv, hu), tot))
    h, hv, hu = _T(n0, n1, n2)
    return _drag(*_post(h, hu, hv), g["manning"], dt), smx, smy


def _eig(z):
    """Roe eigenstructure (u_n, u_t, c, any) of neighbouring cells."""
    n = z["h"].shape[-1]
    a, b = _at(z, 0, n - 1), _at(z, 1, n)
    both = a["wet"] & b["wet"]
    ao = a["wet"] & ~b["wet"] & (b["B"] < a["h"] + a["B"])
    bo = ~a["wet"] & b["wet"] & (a["B"] < b["h"] + b["B"])
    den = torch.where(both, a["s"] + b["s"], torch.ones_like(a["s"]))
    mean = lambda f: torch.where(both, (a["s"] * a[f] + b["s"] * b[f]) / den, torch.where(ao, a[f], b[f]))  # noqa: E731
    c = torch.where(both, torch.sqrt(G * 0.5 * (a["h"] + b["h"]).clamp(min=0.0)), torch.where(ao, a["c"], b["c"]))
    return mean("u"), mean("v"), c, both | ao | bo


def _part(e, d, plus):
    """The part of fluctuation d (mass, normal, transverse) that goes to the high (plus) or low side."""
    u, v, c, on = e
    go = (lambda x: x.clamp(min=0.0)) if plus else (lambda x: x.clamp(max=0.0))  # noqa: E731
    i2 = 0.5 / torch.where(on & (c > 0), c, torch.ones_like(c))
    k1 = go(u - c) * ((u + c) * d[0] - d[1]) * i2
    k3 = go(u + c) * (d[1] - (u - c) * d[0]) * i2
    r = [k1 + k3, k1 * (u - c) + k3 * (u + c), (k1 + k3) * v + go(u) * (d[2] - v * d[0])]
    return [torch.where(on, x, torch.zeros_like(x)) for x in r]


def _unsplit(q, B, g, dt):
    h, hu, hv = q
    rx, ry = dt / g["dx"], dt / g["dy"]
    zx, zy = _cell(h, hu, hv, B), _cell(*_T(h, hv, hu, B))
    ax = _limited(zx, rx)
    ay = _limited(zy, ry)
    # fluctuations entering each cell, first order and second order
    S = lambda a: [a[1][m][:, :-1] + a[0][m][:, 1:] for m in range(3)]  # noqa: E731
    S2 = lambda a: [(a[1][m] - 2 * a[2][m])[:, :-1] + (a[0][m] + 2 * a[2][m])[:, 1:] for m in range(3)]  # noqa: E731
    Sx, Dx, Sy, Dy = S(ax), S2(ax), S(ay), S2(ay)   # x terms: (ny + 4, nx), y terms: (nx + 4, ny)

    def corrected(z, F, D, r):
        # z: cells of the sweep's frame; D: the other sweep's terms of the cells, in this frame
        e = [x[2:-2, 1:-1] for x in _eig(z)]
        lo, hi = _part(e, [d[:, 1:-2] for d in D], True), _part(e, [d[:, 2:-1] for d in D], False)
        return [F[m][2:-2] - 0.5 * r * (lo[m] + hi[m]) for m in range(3)]

    swap = lambda D: _T(D[0], D[2], D[1])  # noqa: E731
    Gc = corrected(zy, ay[2], swap(Dx), rx)
    Fc = corrected(zx, ax[2], swap(Dy), ry)
    ux = [Sx[m][2:-2] + Fc[m][:, 1:] - Fc[m][:, :-1] for m in range(3)]
    uy = swap([Sy[m][2:-2] + Gc[m][:, 1:] - Gc[m][:, :-1] for m in range(3)])
    new = [x[2:-2, 2:-2] - rx * a - ry * b for x, a, b in zip(q, ux, uy)]
    smx, smy = float(ax[3][2:-2].max()), float(ay[3][2:-2].max())
    return _drag(*_post(*new), g["manning"], dt), smx, smy


def _ghosted(q, bc):
    """Two ghost cells per side: extrapolation (1) or mirror walls (0), x first, then y; q[1] and q[2] are hu and hv."""
    out = []
    for m, a in enumerate(q):
        for d, (lo, hi) in ((1, bc[:2]), (0, bc[2:])):
            n = a.shape[d]
            idx = [1, 0] if lo == 0 else [0, 0]
            jdx = [n - 1, n - 2] if hi == 0 else [n - 1, n - 1]
            normal = m == 2 - d   # hu across x edges, hv across y edges
            A = a.index_select(d, torch.tensor(idx, device=a.device)) * (-1.0 if lo == 0 and normal else 1.0)
            Z = a.index_select(d, torch.tensor(jdx, device=a.device)) * (-1.0 if hi == 0 and normal else 1.0)
            a = torch.cat([A, a, Z], d)
        out.append(a)
    return out


def _sample(grid, xs, ys):
    """Bilinear values of a node grid at the points xs x ys, and where it covers them."""
    v, x0, y0, dx, dy = grid
    v = np.asarray(v, dtype=np.float64)
    axes = []
    for p, o, d, n in ((xs, x0, dx, v.shape[1]), (ys, y0, dy, v.shape[0])):
        f = (p - o) / d
        i = np.clip(np.floor(f).astype(int), 0, n - 2)
        axes.append((i, np.clip(f - i, 0.0, 1.0), (p >= o) & (p <= o + (n - 1) * d)))
    (i, tx, ix), (j, ty, iy) = axes
    i, tx, j, ty = i[None, :], tx[None, :], j[:, None], ty[:, None]
    a = v[j, i] + tx * (v[j, i + 1] - v[j, i])
    b = v[j + 1, i] + tx * (v[j + 1, i + 1] - v[j + 1, i])
    return a + ty * (b - a), iy[:, None] & ix[None, :]


def _exact_grid(case, seed):
    w = _grid_workload(case, seed)
    cfg = w["cfg"]
    nx, ny = case["nx"], case["ny"]
    xs = cfg["x0"] + (np.arange(nx) + 0.5) * cfg["dx"]
    ys = cfg["y0"] + (np.arange(ny) + 0.5) * cfg["dy"]

    def on(grid):
        v, inside = _sample(grid, xs, ys)
        return torch.from_numpy(np.where(inside, v, 0.0)).cuda()

    B0 = on(w["topo"][0])
    eta = on(w["eta"][0][1:]) if w["eta"] else torch.zeros_like(B0)
    B = B0 + (on(w["uplift"][0][1:]) if w["uplift"] else 0.0)
    h = torch.clamp(eta - B0, min=0.0)
    hu, hv = torch.zeros_like(h), torch.zeros_like(h)
    if w.get("uv"):
        s, u, v, *at = w["uv"][0]
        wet = h >= DRYTOL
        hu, hv = (torch.where(wet, h * on((a, *at)), torch.zeros_like(h)) for a in (u, v))
    unit = cfg["earth_radius"] * math.pi / 180.0 if case["lonlat"] else 1.0
    g = dict(nx=nx, ny=ny, dx=cfg["dx"] * unit, dy=cfg["dy"] * unit, lonlat=case["lonlat"], y0=cfg["y0"],
             ddy=cfg["dy"], manning=case["manning"])
    step = _unsplit if case["scheme"] == "unsplit" else _split
    kap, ced = _sphere(g)
    k, c = kap[2:-2, None], ced[2:-2]
    z = _cell(h, hu, hv, B)
    rate = max(float(((z["u"].abs() + z["c"]) / k).max()) / g["dx"],
               float(((z["v"].abs() + z["c"]) * torch.maximum(c[:-1], c[1:])[:, None] / k).max()) / g["dy"])
    q, t = [h, hu, hv], 0.0
    Bg = _ghosted([B], cfg["bc"])[0]
    for _ in range(case["steps"]):
        dt = cfg["cfl_desired"] / rate
        full = _ghosted(q, cfg["bc"])
        new, sx, sy = step(full, Bg, g, dt)
        rate = max(sx / g["dx"], sy / g["dy"])
        if dt * rate > cfg["cfl_max"]:   # taken again from the same state
            dt = cfg["cfl_desired"] / rate
            new, sx, sy = step(full, Bg, g, dt)
            rate = max(sx / g["dx"], sy / g["dy"])
        q, t = list(new), t + dt
    if case["prec"] == "f32":   # the FP32 form keeps the surface in place of the depth
        q[0] = q[0] + B
    return dict(t=t, q=q)


def exact(case, seed):
    kind = case["kind"]
    if kind == "grid":
        return _exact_grid(case, seed)
    if kind == "block":
        q0, hu, hv, B = (a.double() for a in _block_state(case, seed))
        g = dict(nx=case["nx"], ny=case["ny"], dx=BLOCK_DX, dy=BLOCK_DX, lonlat=False, manning=0.0)
        bc = [W.BC_EXTRAP] * 2 + [W.BC_WALL] * 2
        h = q0 - B if case["prec"] == "f32" else q0
        q, sx, sy = _split(_ghosted([h, hu, hv], bc), _ghosted([B], bc)[0], g, _block_dt())
        q = list(q)
        if case["prec"] == "f32":
            q[0] = q[0] + B
        return dict(speeds=[sx, sy], q=q)
    if kind in ("amr", "ensemble"):
        return None   # a whole hierarchy with its regrids: no plain counterpart
    theta, x, target, mask = (torch.from_numpy(np.asarray(a, dtype=np.float64)).cuda() for a in _cnn_inputs(case, seed))
    theta.requires_grad_(kind == "grad")
    a, o = x, 0
    for ci, co, kk in ((5, 16, 3), (16, 16, 3), (16, 16, 3), (16, 1, 1)):
        wgt = theta[o:o + co * ci * kk * kk].reshape(co, ci, kk, kk)
        o += co * ci * kk * kk
        a = torch.nn.functional.conv2d(a, wgt, theta[o:o + co], padding=kk // 2)
        a = a.relu() if co > 1 else a
        o += co
    z = a[:, 0]
    if kind == "logits":
        return z
    loss = (torch.nn.functional.binary_cross_entropy_with_logits(z, target, reduction="none") * mask).sum() / mask.sum()
    loss.backward()
    return dict(loss=loss.detach(), grad=theta.grad)
