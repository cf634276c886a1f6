"""The update's tiles and the launches around them at the sizes where they can
go wrong: strips and row segments that end one cell before a patch does, a few
cells, levels of more tiles than the last CTA counts, grids in the caller's memory,
layers whose images do not fill their tiles.

FP64 repeats the oracle's operations in its order, so its fields equal the
oracle's bits.  The FP32 update's result for a cell depends on the cells around it
only, not on the tile that holds them, so every cut of a level gives the same bits.
"""
import numpy as np
import pytest

import oracle
from oracle import cnn as ocnn
from paper_1901_06798_gb300 import workloads as W

pytestmark = pytest.mark.gpu

F32P_ETA = 1e-4   # metres: the FP32 perturbation form against the FP64 oracle
FIELDS = ("eta", "hu", "hv")


def _hump(nx, ny, **kw):
    """The 2 km basin's hump on nx x ny cells, walls and open edges."""
    w = W.hump200()
    cfg = dict(w["cfg"], nx=nx, ny=ny, dx=2000.0 / nx, dy=2000.0 / ny, bc=[0, 1, 1, 0], **kw)
    return dict(w, cfg=cfg)


def _run(w, prec, steps, tuning=None, bulk=0):
    from paper_1901_06798_gb300 import binding
    g = W.load(binding.Tsunami(w["cfg"], precision=prec), w)
    if tuning:
        g.set_tuning(*tuning)
    if bulk:
        g.set_bulk_copies(1)
    g.step(steps)
    out = {f: g.level_array(0, 1, f) for f in FIELDS}
    gauges = g.read_gauges()
    g.close()
    return out, gauges


# 5: 1600 tiles, a launch of its own ends the step; 6: 1156 tiles, the last CTA does;
# 61: strips and segments that end one cell before the patch's neighbours begin
@pytest.mark.parametrize("lonlat", [False, True])
@pytest.mark.parametrize("tile", [5, 6, 61, 62])
def test_level1_tiles_same_bits(tile, lonlat):
    def case(t):
        w = W.shelf(n=200, dx=2000.0)
        w = dict(w, cfg=dict(w["cfg"], level1_tile=t))
        return W.lonlat(w) if lonlat else w
    one, _ = _run(case(0), 1, 12)
    for tuning, bulk in ((None, 0), ((128, 2), 0), ((64, 59), 0), (None, 1)):
        got, _ = _run(case(tile), 1, 12, tuning, bulk)
        for f in FIELDS:
            assert np.array_equal(got[f], one[f]), (f, tuning, bulk)
    w = case(tile)
    o = W.load(oracle.Oracle(w["cfg"]), w)
    o.step(12)
    got, (tg, eg) = _run(w, 0, 12)
    to, eo = o.read_gauges()
    assert np.array_equal(tg, to) and np.array_equal(eg, eo)
    for f in FIELDS:
        assert np.array_equal(got[f], o.level_array(0, 1, f)), f
    wet = o.level_array(0, 1, "h") > 0
    assert np.abs(one["eta"] - o.level_array(0, 1, "eta"))[wet].max() <= F32P_ETA


@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 2), (59, 32), (60, 33), (61, 2), (121, 7), (180, 127)])
def test_grid_sizes_match_oracle(nx, ny):
    w = _hump(nx, ny)
    o = W.load(oracle.Oracle(w["cfg"]), w)
    o.step(15)
    ref = {f: o.level_array(0, 1, f) for f in FIELDS}
    for tuning in (None, (64, 3), (256, 64)):
        got, _ = _run(w, 0, 15, tuning)
        for f in FIELDS:
            assert np.array_equal(got[f], ref[f]), (f, tuning)
    first = None
    for tuning in (None, (32, 1), (64, 7), (128, 124), (256, 31)):
        got, _ = _run(w, 1, 15, tuning)
        first = first or got
        for f in FIELDS:
            assert np.array_equal(got[f], first[f]), (f, tuning)
    assert np.abs(first["eta"] - ref["eta"]).max() <= F32P_ETA


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nx,ny", [(2, 2), (5, 3), (61, 45), (200, 129)])
def test_noalloc_grids_match_context_bits(nx, ny, prec):
    """Two steps of a grid in the caller's memory at an odd pitch, speeds to pageable
    memory: the context's bits, and the speeds of a second call on the same state."""
    import torch
    from paper_1901_06798_gb300 import binding
    dt = 0.1
    w = _hump(nx, ny, dt_max=dt)
    ctx = W.load(binding.Tsunami(w["cfg"], precision=prec), dict(w, gauges=np.zeros((0, 2))))
    (_, a0), = ctx.patches(0, 1)
    ctx.step(2)
    (_, a2), = ctx.patches(0, 1)
    ctx.close()
    pitch = nx + 9
    fs = pitch * (ny + 4) + 3
    host = np.zeros(7 * fs, dtype=np.float64 if prec == 0 else np.float32)

    def field(k):
        return host[k * fs:k * fs + pitch * (ny + 4)].reshape(ny + 4, pitch)[2:ny + 2, 2:nx + 2]
    for k, v in ((0, a0["h"] if prec == 0 else a0["h"] + a0["B"]), (1, a0["hu"]), (2, a0["hv"]), (6, a0["B"])):
        field(k)[:] = v
    dev = torch.from_numpy(host).cuda()
    c = w["cfg"]
    st = torch.cuda.current_stream().cuda_stream
    speeds = []
    for cur in (0, 0, 1):
        rc, s = binding.tsu_grid_step_noalloc(prec, dev.data_ptr(), nx, ny, pitch, fs, cur, c["dx"], c["dy"], dt, c["g"],
                                              c["drytol"], c["bc"], st)
        assert rc == binding.TSU_OK
        speeds.append(tuple(s))
    assert speeds[0] == speeds[1]
    host[:] = dev.cpu().numpy()
    B = field(6).astype(np.float64)
    h = field(0).astype(np.float64) - (B if prec == 1 else 0.0)
    for mine, f in ((h, "h"), (field(1), "hu"), (field(2), "hv")):
        assert np.array_equal(mine.astype(np.float64), a2[f].astype(np.float64)), f


# the tolerances that the predictor's tests have: 1e-4 of the largest value
@pytest.mark.parametrize("n,h,w", [(1, 1, 1), (3, 8, 32), (2, 9, 33), (1, 7, 65), (17, 3, 5)])
def test_predictor_on_uneven_images(n, h, w):
    from paper_1901_06798_gb300 import binding
    theta = ocnn.init_params(5)
    rng = np.random.default_rng(1000 * n + 10 * h + w)
    x = rng.normal(size=(n, ocnn.C_IN, h, w))
    t = (rng.random((n, h, w)) < 0.25).astype(float)
    m = np.ones((n, h, w))
    ref, _ = ocnn.forward(theta, x)
    scale = np.abs(ref).max()
    assert np.abs(binding.cnn_forward(theta, x, fp16=False) - ref).max() <= 1e-4 * scale
    assert np.abs(binding.cnn_forward(theta, x, fp16=True) - ref).max() <= 2e-2 * scale
    loss_ref, g_ref = ocnn.backward(theta, x, t, m)
    loss, g = binding.cnn_loss_grad(theta, x, t, m)
    assert loss == pytest.approx(loss_ref, rel=1e-5)
    assert np.abs(g - g_ref).max() <= 1e-4 * np.abs(g_ref).max()


@pytest.mark.parametrize("nx,ny", [(1, 1), (127, 33), (129, 31), (300, 5)])
def test_rasters_of_odd_sizes_match_oracle(nx, ny):
    w = W.shelf(n=96, dx=2000.0)
    cfg = dict(w["cfg"], num_levels=2, ratios=[4], regrid_interval=3, flag_eta_tol=0.05, patch_max=32)
    w = dict(w, cfg=cfg)
    from paper_1901_06798_gb300 import binding
    o = W.load(oracle.Oracle(cfg), w)
    g = W.load(binding.Tsunami(cfg, precision=0), w)
    o.step(4)
    g.step(4)
    L = cfg["nx"] * cfg["dx"]
    # (the last points lie outside the domain)
    for lev in (0, 1, 2):
        args = (0, lev, "eta", nx, ny, 37.0, 53.0, 1.05 * L / nx, 1.02 * L / ny)
        assert np.array_equal(o.read_field(*args), g.read_field(*args), equal_nan=True), lev
