"""Grids a few cells thick: lines that would leave most of a tile unused stream
instead (the range of a tiled line is the line itself, a streamed one is at
least 24 positions), small ones keep their tiles, and both give the same
bits."""
import numpy as np
import pytest

from paper_1206_0919_gb300 import shasta as S
from paper_1206_0919_gb300 import workloads as W
from oracle import oracle as OR
from gpu_util import oracle, require_gpu

pytestmark = pytest.mark.gpu


def run(shape, U, tune, **kw):
    with S.Solver(shape, autotune=tune, **kw) as s:
        s.set_conserved(U)
        s.step(2)
        return s.get_conserved(), [r for _, r in s.tuning()]


@pytest.mark.parametrize("precision", ["fp32", "mixed", "mixed_fp64"])
@pytest.mark.parametrize("shape,thin", [((512, 512, 4), 2), ((4, 512, 512), 0), ((512, 8, 512), 1), ((24, 24, 4), None),
                                        ((1, 40, 40), None)])
def test_thin_grids(monkeypatch, precision, shape, thin):
    require_gpu()
    pr = W.random_state(shape, seed=3, vmax=0.5)
    U = oracle().prim2cons(OR.params(shape), *pr.as_list())
    monkeypatch.setenv("SHASTA_TILE", "off")
    ref, _ = run(shape, U, False, precision=precision)
    monkeypatch.setenv("SHASTA_TILE", "")
    for tune in (False, True):
        got, ranges = run(shape, U, tune, precision=precision)
        for a, b in zip(ref, got):
            assert np.array_equal(a, b)
        if not tune and thin is not None:
            assert ranges[thin] >= 24 > shape[thin]
        if thin is None:
            assert all(r <= n for r, n in zip(ranges, shape))


@pytest.mark.parametrize("shape,axis,tile", [((300, 20, 24), 0, 100), ((430, 9, 12), 0, 144), ((20, 160, 24), 1, 80),
                                             ((24, 20, 230), 2, 115)])
def test_small_grids_show_their_tiles(monkeypatch, shape, axis, tile):
    """The range of a tiled axis is the length of its tiles (a line in equal
    parts), which no streamed choice is: those are whole lines or the positions
    per resident warp, 24 on grids this small."""
    require_gpu()
    pr = W.random_state(shape, seed=5, vmax=0.5)
    U = oracle().prim2cons(OR.params(shape), *pr.as_list())
    res = []
    for env in ("", "off"):
        monkeypatch.setenv("SHASTA_TILE", env)
        for tune in (False, True):
            res.append(run(shape, U, tune))
            assert (res[-1][1][axis] == tile) == (env == ""), (env, tune, res[-1][1])
    for got, _ in res[1:]:
        for a, b in zip(res[0][0], got):
            assert np.array_equal(a, b)
