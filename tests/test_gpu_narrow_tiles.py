"""FP64 tiles of at most 28 columns, whose x sweep takes two rows of a warp: widths on both
sides of the line, odd and even numbers of rows, strips that end in a narrow tile.  The
fields are the oracle's bits."""
import numpy as np
import pytest

import oracle
from paper_1901_06798_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FIELDS = ("h", "hu", "hv")


def _check(w, steps, tuning):
    from paper_1901_06798_gb300 import binding
    o = W.load(oracle.Oracle(w["cfg"]), w)
    o.step(steps)
    for tn in tuning:
        g = W.load(binding.Tsunami(w["cfg"], precision=0), w)
        if tn:
            g.set_tuning(*tn)
        g.step(steps)
        assert g.stats()["t"] == o.stats()["t"]
        for f in FIELDS:
            assert np.array_equal(g.level_array(0, 1, f), o.level_array(0, 1, f)), (f, tn)
        g.close()


@pytest.mark.parametrize("lonlat", [False, True])
@pytest.mark.parametrize("tile", [1, 13, 27, 28, 29])
def test_patches_of_few_columns(tile, lonlat):
    """The shelf with its beach, moving water everywhere, drag."""
    w = W.shelf(n=58, dx=8000.0)
    L = 58 * 8000.0
    x = np.linspace(0.0, 1.0, 59)
    u = 0.05 * np.sin(9.0 * x)[None, :] * np.cos(7.0 * x)[:, None]
    w = dict(w, cfg=dict(w["cfg"], level1_tile=tile, manning_n=0.025), uv=[(0, u, u.T.copy(), 0.0, 0.0, L / 58, L / 58)])
    _check(W.lonlat(w) if lonlat else w, 8, (None, (64, 5), (256, 3)))


@pytest.mark.parametrize("nx,ny", [(28, 3), (29, 8), (88, 41), (89, 40), (31, 75)])
def test_grids_that_end_in_a_narrow_strip(nx, ny):
    w = W.hump200()
    cfg = dict(w["cfg"], nx=nx, ny=ny, dx=2000.0 / nx, dy=2000.0 / ny, bc=[0, 1, 1, 0])
    _check(dict(w, cfg=cfg), 15, (None, (64, 3), (128, 7)))
