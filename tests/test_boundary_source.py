"""Ghost cells of the physical boundaries (csrc/boundary.h): every one takes its
values from a cell of the domain, also where the domain is one cell wide and the
image of the second ghost cell lies past the other edge.

On the CPU the rule is compiled as it stands and compared with reflections done one
at a time.  On the GPU a step of a one-cell-wide grid, its ghost rings full of
other values, equals the middle of the same step on the grid unfolded to five cells.
"""
import ctypes
import itertools
import os
import subprocess

import numpy as np
import pytest

from paper_1901_06798_gb300 import workloads as W

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_06798_gb300", "csrc")
WALL, EXTRAP = W.BC_WALL, W.BC_EXTRAP


def _source(i, n, lo, hi):
    """(cell, sign of the normal momentum) of index i."""
    sign = 1
    while not 0 <= i < n:
        if i < 0:
            i, sign = (-1 - i, -sign) if lo == WALL else (0, sign)
        else:
            i, sign = (2 * n - 1 - i, -sign) if hi == WALL else (n - 1, sign)
    return i, sign


def test_sources_lie_in_the_domain(tmp_path):
    src = tmp_path / "b.cpp"
    src.write_text('#include "boundary.h"\n'
                   'extern "C" int f(int I, int n, int lo, int hi, int *src, int *flip) {\n'
                   '    bool fl; int out = tsu::boundary_source(I, n, lo, hi, *src, fl); *flip = fl; return out; }\n')
    so = tmp_path / "b.so"
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    f = ctypes.CDLL(str(so)).f
    for n, lo, hi in itertools.product((1, 2, 3, 60), (WALL, EXTRAP), (WALL, EXTRAP)):
        for i in range(-2, n + 2):
            s, fl = ctypes.c_int(), ctypes.c_int()
            out = f(i, n, lo, hi, ctypes.byref(s), ctypes.byref(fl))
            assert bool(out) == (not 0 <= i < n)
            assert 0 <= s.value < n and (s.value, -1 if fl.value else 1) == _source(i, n, lo, hi), (n, lo, hi, i)


def _step(prec, q, bc, junk):
    """Interior (q0, hu, hv) and the speeds after one step of the grid q = (q0, hu, hv, B)."""
    import torch
    from paper_1901_06798_gb300 import binding
    ny, nx = q[0].shape
    block = np.full((7, ny + 4, nx + 4), junk, dtype=np.float64 if prec == 0 else np.float32)
    for f, a in zip((0, 1, 2, 6), q):
        block[f, 2:-2, 2:-2] = a
    dev = torch.from_numpy(block).cuda()
    rc, speeds = binding.tsu_grid_step_noalloc(prec, dev.data_ptr(), nx, ny, nx + 4, (nx + 4) * (ny + 4), 0, 10.0, 10.0, 0.2,
                                               9.81, 1e-3, bc, torch.cuda.current_stream().cuda_stream)
    assert rc == binding.TSU_OK
    return dev.cpu().numpy()[3:6, 2:-2, 2:-2], tuple(speeds)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 70), (70, 1), (1, 2)])
@pytest.mark.parametrize("bc", [(WALL,) * 4, (WALL, EXTRAP, EXTRAP, WALL), (EXTRAP, WALL, WALL, EXTRAP), (EXTRAP,) * 4])
def test_one_cell_wide_grids(nx, ny, bc, prec):
    rng = np.random.default_rng(100 * nx + ny)
    B = -20.0 + rng.random((ny, nx))
    h = -B + 0.5 * rng.random((ny, nx))
    q = [h if prec == 0 else h + B, 20.0 * rng.random((ny, nx)) - 5.0, 20.0 * rng.random((ny, nx)) - 5.0, B]
    got, speeds = _step(prec, q, bc, 3.0)
    again, speeds2 = _step(prec, q, bc, -77.0)
    assert np.array_equal(got, again) and speeds == speeds2
    assert np.isfinite(got).all() and 10.0 < min(speeds) and max(speeds) < 20.0
    # unfolded: two more cells on each side of an axis of one cell, from the rule
    ix = [_source(i, nx, *bc[:2]) for i in (range(-2, 3) if nx == 1 else range(nx))]
    iy = [_source(j, ny, *bc[2:]) for j in (range(-2, 3) if ny == 1 else range(ny))]
    wide = [a[np.ix_([j for j, _ in iy], [i for i, _ in ix])] for a in q]
    wide[1] = wide[1] * np.array([s for _, s in ix])[None, :]
    wide[2] = wide[2] * np.array([s for _, s in iy])[:, None]
    ref, _ = _step(prec, wide, bc, 0.0)
    if nx == 1:
        ref = ref[:, :, 2:3]
    if ny == 1:
        ref = ref[:, 2:3, :]
    assert np.array_equal(got, ref)
