"""CFL retakes (Sec. 2.2) where their launch can go wrong: more tiles than the FP32
retake's CTAs (608), so that a CTA takes several; more than the last CTA of the update
counts (1216), so that a launch of its own checks the step and the retake's last CTA
ends it; scenarios of which only some are retaken, whose time and gauge samples wait
for the others.

FP64 repeats the oracle's bits.  FP32 gives the same bits for every cut of the grid
and for a scenario alone.
"""
import numpy as np
import pytest

import oracle
from paper_1901_06798_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 24
FIELDS = ("h", "hu", "hv")


def _channel(ny, transverse=0):
    """The stepped channel ny cells wide, its velocities varying along y, with gauges."""
    w = W.stepped_channel(3, ny=ny)
    k = 1.0 + 0.2 * np.cos(0.05 * np.arange(ny + 1))[:, None]
    uv = [(s, u * k, v * k, *g) for s, u, v, *g in w["uv"]]
    gauges = np.array([[7.3, 0.4 * ny], [22.1, 0.9 * ny], [38.6, 1.2]])
    return dict(w, cfg=dict(w["cfg"], transverse=transverse), uv=uv, gauges=gauges)


def _several(w):
    """Three scenarios in the channel: as it is, still water, and slower."""
    still = lambda a: np.zeros_like(a)   # noqa: E731
    eta = [(s, f(e), *g) for s, f in ((0, lambda a: a), (1, still), (2, lambda a: 0.5 * a)) for _, e, *g in w["eta"]]
    uv = [(s, f(u), f(v), *g) for s, f in ((0, lambda a: a), (1, still), (2, lambda a: 0.3 * a)) for _, u, v, *g in w["uv"]]
    return dict(w, cfg=dict(w["cfg"], n_scenarios=3), eta=eta, uv=uv)


def _one(w, s):
    return dict(w, cfg=dict(w["cfg"], n_scenarios=1), eta=[(0, *e[1:]) for e in w["eta"] if e[0] == s],
                uv=[(0, *e[1:]) for e in w["uv"] if e[0] == s])


def _run(w, prec, tuning=None, by_level=False):
    from paper_1901_06798_gb300 import binding
    g = W.load(binding.Tsunami(w["cfg"], precision=prec), w)
    if tuning:
        g.set_tuning(*tuning)
    t = [np.array(g.step(1, allow_cfl=True)) for _ in range(STEPS - 10)]   # captured steps of both parities
    t.append(np.array(g.step(10, allow_cfl=True)))
    n = w["cfg"].get("n_scenarios", 1)
    out = dict(t=np.array(t), gauges=g.read_gauges(), stats=[g.stats(s) for s in range(n)],
               q=[[g.level_array(s, 1, f) for f in FIELDS] for s in range(n)])
    g.close()
    return out


def _oracle(w):
    o = W.load(oracle.Oracle(w["cfg"]), w)
    t = [np.array(o.step(1)) for _ in range(STEPS - 10)]
    t.append(np.array(o.step(10)))
    n = w["cfg"].get("n_scenarios", 1)
    return dict(t=np.array(t), gauges=o.read_gauges(), stats=[o.stats(s) for s in range(n)],
                q=[[o.level_array(s, 1, f) for f in FIELDS] for s in range(n)])


def _same(a, b):
    assert np.array_equal(a["t"], b["t"])
    for x, y in zip(a["gauges"], b["gauges"]):
        assert np.array_equal(x, y, equal_nan=True)
    for x, y in zip(a["stats"], b["stats"]):
        for k in ("cfl_retakes", "cfl_violations", "cell_updates"):
            assert x[k] == y[k], k
    for x, y in zip(a["q"], b["q"]):
        for f, p, q in zip(FIELDS, x, y):
            assert np.array_equal(p, q), f


# 650: more tiles of 2 rows than the FP32 retake's CTAs; 1300: more than are counted
@pytest.mark.parametrize("tiles", [650, 1300])
def test_retakes_on_many_tiles(tiles):
    w = _channel(2 * tiles)
    ref = _oracle(w)
    assert ref["stats"][0]["cfl_retakes"] >= 2
    _same(_run(w, 0, (128, 2)), ref)
    one = _run(w, 1, (128, 60))   # an item per CTA, the last CTA counts
    assert one["stats"][0]["cfl_retakes"] >= 2
    _same(_run(w, 1, (128, 2)), one)
    _same(_run(w, 1), one)


@pytest.mark.parametrize("transverse", [0, 1])
@pytest.mark.parametrize("ny", [4, 900])
def test_retakes_of_some_scenarios(ny, transverse):
    """900: 1350 tiles of 2 rows over the three scenarios."""
    w = _several(_channel(ny, transverse))
    ref = _oracle(w)
    retakes = [s["cfl_retakes"] for s in ref["stats"]]
    assert retakes[0] >= 1 and retakes[1] == 0 and len(set(retakes)) >= 2
    for tuning in (None, (128, 2)):
        _same(_run(w, 0, tuning), ref)
        got = _run(w, 1, tuning)
        assert got["stats"][0]["cfl_retakes"] >= 1 and got["stats"][1]["cfl_retakes"] == 0
        for s in range(3):
            alone = _run(_one(w, s), 1, tuning)
            assert np.array_equal(got["t"][:, s], alone["t"][:, 0])
            for k in ("cfl_retakes", "cfl_violations", "cell_updates"):
                assert got["stats"][s][k] == alone["stats"][0][k], (s, k)
            for p, q in zip(got["q"][s], alone["q"][0]):
                assert np.array_equal(p, q), s
            (tg, eg), (ta, ea) = got["gauges"], alone["gauges"]
            assert np.array_equal(tg[:, s], ta[:, 0]) and np.array_equal(eg[:, s], ea[:, 0], equal_nan=True)
