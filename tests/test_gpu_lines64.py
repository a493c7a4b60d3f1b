"""FP64 whole-line sweeps against the FP64 streaming sweeps, bit for bit.

Lines of 3 cells (the shortest the mirrored reads allow) up to the longest
that fit a block, lines per block that leave the last block partly empty,
more cells than a block has threads, every boundary rule and equation of
state.  The states mix ordinary cells with what leaves the fast forms: cells
at rest, momenta down to 1e-305, |M| > E (clamped and counted), E <= 0, and energies scaled by powers
of ten down to 1e-130 and up to 1e130 (their squares leave the range in which
the short quotient and root hold)."""
import numpy as np
import pytest

from paper_1206_0919_gb300 import shasta as S
from paper_1206_0919_gb300 import workloads as W
from oracle import oracle as OR
from gpu_util import oracle, require_gpu

pytestmark = pytest.mark.gpu

TABLE = np.arange(4001) * 0.01 / 3.0


def state(shape, seed, wild):
    pr = W.random_state(shape, seed=seed, vmax=0.6, e_range=(0.3, 3.0))
    U = [u.copy() for u in oracle().prim2cons(OR.params(shape), *pr.as_list())]
    rng = np.random.default_rng(seed)
    rest = rng.random(U[0].shape) < 0.3
    for k in (1, 2, 3):
        U[k][rest] = 0.0
    tail = rng.random(U[0].shape) < 0.2  # momenta of every magnitude, as far out in a front
    for k in (1, 2, 3):
        U[k][tail] *= 10.0 ** -rng.uniform(0, 305, U[0].shape)[tail]
    U[1].flat[5] = 1.5 * U[0].flat[5]
    if wild:
        far = rng.random(U[0].shape) < 0.2
        s = np.where(far, 10.0 ** rng.integers(-130, 131, U[0].shape), 1.0)
        U = [u * s for u in U]
        U[0].flat[7] = 0.0
        U[0].flat[-3] = -1e-3
    return U


def run(monkeypatch, lines, shape, U, steps, **kw):
    if lines:
        monkeypatch.setenv("SHASTA_LINES", lines)
    else:
        monkeypatch.delenv("SHASTA_LINES", raising=False)
    with S.Solver(shape, precision="fp64", check_input=False, autotune=False, **kw) as s:
        s.set_conserved(U)
        s.step(steps)
        return s.get_conserved(), s.counters()


@pytest.mark.parametrize("bc", ["reflect", "periodic", "frozen"])
@pytest.mark.parametrize("eos", ["ideal", "bag", "table"])
def test_lines_match_streaming_bitwise(monkeypatch, eos, bc):
    require_gpu()
    kw = dict(eos=eos, bc=bc)
    if eos == "table":
        kw.update(table=TABLE, table_de=0.01)
    for i, shape in enumerate([(3, 4, 5), (2, 33, 7), (64, 31, 9), (40, 65, 3), (170, 13, 16), (5, 874, 3),
                               (875, 3, 4)]):
        for wild in (False, True):
            U = state(shape, 10 * i + wild, wild and eos != "table")
            steps = 1 if wild else 7
            ref = run(monkeypatch, "off", shape, U, steps, **kw)
            for lines in (None, "1", "3"):
                got = run(monkeypatch, lines, shape, U, steps, **kw)
                assert got[1] == ref[1] > 0, (shape, wild, lines)
                for a, b in zip(ref[0], got[0]):
                    assert np.array_equal(a, b, equal_nan=True), (shape, wild, lines)


@pytest.mark.parametrize("de", [0.01, 2.0 ** -40, 0.3])
def test_table_index_and_fraction_at_the_nodes(monkeypatch, de):
    """The index and fraction taken from the bit pattern give what the
    conversions give: energies on, one ulp below and above a table's nodes,
    below the first interval's end, above the table and far above it."""
    require_gpu()
    table = np.arange(40) * de * 0.25
    k = np.arange(1, 60) * de
    e = np.concatenate([k, np.nextafter(k, 0), np.nextafter(k, 1e9), de * 10.0 ** -np.arange(1, 20), de * 2.0 ** np.arange(5, 40)])
    shape = (e.size, 4, 3)
    U = [np.broadcast_to(e, (3, 4, e.size)).copy() for _ in range(5)]
    for j, f in enumerate((0.0, 0.3, -0.2)):
        U[1 + j] = f * U[0] * (np.arange(4) % 2)[None, :, None]
    kw = dict(eos="table", table=table, table_de=de)
    ref = run(monkeypatch, "off", shape, U, 3, **kw)
    got = run(monkeypatch, None, shape, U, 3, **kw)
    assert got[1] == ref[1]
    for a, b in zip(ref[0], got[0]):
        assert np.array_equal(a, b, equal_nan=True)
