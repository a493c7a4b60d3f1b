"""Tiled sweeps against the streaming sweeps, bit for bit.

Every tile shape (cells per lane, lines per warp) is forced on grids whose
lines end inside the first lane group, at a tile's last own cell, one past it,
and in a second and third tile, with line counts that leave tiles partly
empty, for every boundary rule, equation of state and single-precision
recovery; a cell with |M| > E makes the clamped path run and be counted."""
import numpy as np
import pytest

from paper_1206_0919_gb300 import shasta as S
from paper_1206_0919_gb300 import workloads as W
from oracle import oracle as OR
from gpu_util import oracle, require_gpu

pytestmark = pytest.mark.gpu

OWN = [52, 68, 84, 100, 116, 132, 148, 180, 212, 244, 276]  # own positions of each tile shape
TABLE = np.arange(4001) * 0.01 / 3.0


def run(monkeypatch, tile, shape, U, **kw):
    monkeypatch.setenv("SHASTA_TILE", tile)
    with S.Solver(shape, check_input=False, **kw) as s:
        s.set_conserved(U)
        s.step(7)  # every axis order; six steps as one graph
        return s.get_conserved(), s.counters(), [r for _, r in s.tuning()]


@pytest.mark.parametrize("bc", ["reflect", "periodic", "frozen"])
@pytest.mark.parametrize("precision,eos", [("fp32", "ideal"), ("fp32", "bag"), ("fp32", "table"),
                                           ("mixed", "ideal"), ("mixed", "bag"),
                                           ("mixed_fp64", "ideal"), ("mixed_fp64", "bag")])
def test_tiles_match_streaming_bitwise(monkeypatch, precision, eos, bc):
    require_gpu()
    kw = dict(precision=precision, eos=eos, bc=bc)
    if eos == "table":
        kw.update(table=TABLE, table_de=0.01)
    for i, own in enumerate(OWN):
        for shape in ((own, 5, 9), (9, own + 1, 3), (3, 17, own), (own + 1, 2 * own + 3, 2)):
            pr = W.random_state(shape, seed=i + sum(shape), vmax=0.6, e_range=(0.3, 3.0))
            U = oracle().prim2cons(OR.params(shape), *pr.as_list())
            U[1][-1, -1, -2] = 1.5 * U[0][-1, -1, -2]
            ref = run(monkeypatch, "off", shape, U, **kw)
            got = run(monkeypatch, str(i), shape, U, **kw)
            assert got[1] == ref[1] > 0, (i, shape)
            for a, b in zip(ref[0], got[0]):
                assert np.array_equal(a, b), (i, shape)


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 33, 1), (5, 3, 2), (37, 21, 13), (131, 97, 20)])
def test_small_grids_take_tiles(monkeypatch, shape):
    """The default choice on small grids is the tiled sweep (at most a tile's
    own positions per range), with the streaming sweep's results."""
    require_gpu()
    pr = W.random_state(shape, seed=3, vmax=0.6)
    U = oracle().prim2cons(OR.params(shape), *pr.as_list())
    ref = run(monkeypatch, "off", shape, U)
    got = run(monkeypatch, "", shape, U)
    assert all(r <= n for r, n in zip(got[2], shape))
    for a, b in zip(ref[0], got[0]):
        assert np.array_equal(a, b)


BATCH = [((40, 36, 28), "reflect", "ideal"), ((33, 20, 48), "periodic", "bag"), ((24, 40, 16), "frozen", "ideal"),
         ((64, 64, 64), "reflect", "bag"), ((5, 3, 2), "reflect", "ideal"), ((1, 33, 1), "frozen", "bag"),
         ((48, 48, 48), "reflect", "ideal"), ((17, 9, 30), "periodic", "ideal"), ((70, 31, 9), "reflect", "bag")]


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("count", [1, 2, 7, 8, 9])
def test_small_batches_by_event_match_streaming_bitwise(monkeypatch, precision, count):
    """Up to eight small events take tiled launches of their own, more the
    shared streaming launches: the same states and clamp counts, with events at
    different phases, through graphs and single steps, and after a removal."""
    require_gpu()
    res = []
    for tile in ("off", ""):
        monkeypatch.setenv("SHASTA_TILE", tile)
        with S.Batch(600_000, precision=precision, check_input=False) as b:
            ids = []
            for i, (shape, bc, eos) in enumerate(BATCH[:count]):
                pr = W.random_state(shape, seed=40 + i, vmax=0.6, e_range=(0.3, 3.0))
                U = oracle().prim2cons(OR.params(shape), *pr.as_list())
                U[1].flat[-1] = 1.5 * U[0].flat[-1]
                ids.append(b.add_conserved(shape, U, bc=bc, eos=eos))
                if i == 1:
                    b.step(2)
            b.step(7)
            if count > 2:
                b.remove(ids.pop(1))
            b.step(8)
            res.append([(b.get_conserved(e), b.counters(e), b.steps_done(e)) for e in ids])
    for (ua, ca, sa), (ub, cb, sb) in zip(*res):
        assert sa == sb and ca == cb > 0
        for x, y in zip(ua, ub):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("precision,eos", [("fp32", "ideal"), ("fp32", "bag"), ("fp32", "table"), ("mixed", "ideal"),
                                           ("mixed", "bag"), ("mixed_fp64", "ideal")])
@pytest.mark.parametrize("share", [0.002, 0.4])
def test_many_clamped_and_vacuum_cells_bitwise(monkeypatch, precision, eos, share):
    """Warps with a few and with many cells of |M| > E, E = 0 and E < 0, in the
    tiles' own cells, halos and outermost cells: states and counts as streamed,
    also with the atomics of a warp's lanes added up."""
    require_gpu()
    kw = dict(precision=precision, eos=eos)
    if eos == "table":
        kw.update(table=TABLE, table_de=0.01)
    for i, shape in enumerate([(131, 33, 20), (30, 101, 120), (200, 7, 69)]):
        pr = W.random_state(shape, seed=i, vmax=0.6, e_range=(0.3, 3.0))
        U = oracle().prim2cons(OR.params(shape), *pr.as_list())
        pick = np.random.default_rng(i).random(U[0].shape)
        U[2][pick < share] = -2.0 * U[0][pick < share]
        U[0][pick > 1 - share / 4] *= 0.0
        U[0][pick > 1 - share / 8] = -0.1
        ref = run(monkeypatch, "off", shape, U, **kw)
        got = run(monkeypatch, "", shape, U, **kw)
        assert got[1] == ref[1] > share * U[0].size, shape
        for a, b in zip(ref[0], got[0]):
            assert np.array_equal(a, b, equal_nan=True), shape
