"""Input checks, conversions and primitive maps on the GPU at the edges of
their short forms: what the checks refuse (and only that), bit-exact copies
through FP64 and float-rounded copies through FP32 contexts, and the primitive
output against the oracle's maps over all magnitudes."""
import numpy as np
import pytest

from paper_1206_0919_gb300 import shasta as S
from oracle import oracle as OR
from gpu_util import max_rel_err, oracle, require_gpu

pytestmark = pytest.mark.gpu

UP = np.nextafter(1.0, 2.0)
DOWN = np.nextafter(1.0, 0.0)


def physical_cons(E, x, y, z):
    s = (x * x + y * y) + z * z
    return not (E < 0.0 or (s >= E * E and s > 0.0))


@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e60, 2.0 ** -200])
def test_checks_refuse_exactly_the_unphysical_cells(scale):
    """Conserved input is refused exactly where E < 0 or |M| >= E (|M| > 0),
    evaluated in double, for |M| on, one ulp inside and outside, and near the
    light cone; primitives where |v|^2 >= 1, e < 0 or n < 0; NaN and infinity
    always."""
    require_gpu()
    shape = (3, 2, 2)
    one = np.ones((2, 2, 3))
    cons, prim = [], []
    for E in (1.0, 0.0, -0.0, -1.0):
        for m in (0.0, DOWN, 1.0, UP, 1.0 - 2.0 ** -15, 1.0 - 2.0 ** -17, 0.5, 1e-200, 3.0):
            for dirn in ((1, 0, 0), (0, -1, 0), (0.6, 0.0, 0.8), (2 ** -0.5, 2 ** -0.5, 0.0)):
                cons.append((E * scale, *(m * d * scale for d in dirn)))
                prim.append(tuple(m * d for d in dirn))
    with S.Solver(shape, precision="fp64") as s:
        def refused(call):
            try:
                call()
                return False
            except S.ShastaError as e:
                assert e.status == S.EUNPHYSICAL
                return True
        for E, x, y, z in cons:
            U = [one * 2.0 * scale, one * 0, one * 0, one * 0, one.copy()]
            for k, v in enumerate((E, x, y, z)):
                U[k].flat[-1] = v
            assert refused(lambda: s.set_conserved(U)) != physical_cons(E, x, y, z), (E, x, y, z)
        for x, y, z in prim:
            P = [one.copy(), one * 0, one * 0, one * 0, one.copy()]
            for k, v in enumerate((x, y, z)):
                P[1 + k].flat[4] = v
            ok = (x * x + y * y) + z * z < 1.0
            assert refused(lambda: s.set_primitives(*P)) != ok, (x, y, z)
        for k in range(5):
            for v in (np.nan, np.inf, -np.inf):
                U = [one * 2.0, one * 0, one * 0, one * 0, one.copy()]
                U[k].flat[5] = v
                assert refused(lambda: s.set_conserved(U)) and refused(lambda: s.set_primitives(*U))
        for k in (0, 4):
            P = [one.copy(), one * 0, one * 0, one * 0, one.copy()]
            P[k].flat[0] = -1e-300
            assert refused(lambda: s.set_primitives(*P))


@pytest.mark.parametrize("shape", [(1, 1, 1), (7, 5, 3), (32, 32, 1), (64, 33, 17), (128, 128, 65)])
def test_conserved_round_trip(shape):
    """set / get: FP64 contexts return every bit (any subset of the arrays),
    FP32 ones each value rounded to float; one block's cells, one past them,
    and sizes that are converted in several launches."""
    require_gpu()
    nx, ny, nz = shape
    rng = np.random.default_rng(sum(shape))
    U = [rng.normal(size=(nz, ny, nx)) * 10.0 ** rng.integers(-30, 30, (nz, ny, nx)) for _ in range(5)]
    for precision in ("fp64", "fp32"):
        with S.Solver(shape, precision=precision, check_input=False) as s:
            s.set_conserved(U)
            got = s.get_conserved()
            for a, b in zip(U, got):
                ref = a if precision == "fp64" else a.astype(np.float32).astype(np.float64)
                assert np.array_equal(ref, b)
            part = s.get_conserved([None, np.empty_like(U[0]), None, None, np.empty_like(U[0])])
            assert np.array_equal(part[1], got[1]) and np.array_equal(part[4], got[4])
            tot = s.totals()
            for t, b in zip(tot, got):
                assert abs(t - b.sum()) <= 1e-12 * np.abs(b).sum()


@pytest.mark.parametrize("eos", [OR.EOS_IDEAL, OR.EOS_BAG])
@pytest.mark.parametrize("scale", [1.0, 1e-25, 1e25, 1e-140])
def test_primitive_maps_against_oracle(eos, scale):
    """Primitives in and out of an FP64 context against the oracle's maps to
    1e-13 per cell (each is a handful of correctly rounded operations; v up to
    1 - 1e-9 amplifies them by at most gamma^2 of 1e9 in n alone, which is
    compared at v <= 0.99)."""
    require_gpu()
    shape = (33, 9, 7)
    rng = np.random.default_rng(5)
    n = (7, 9, 33)
    e = rng.uniform(0.05, 3.0, n) * scale
    v = rng.normal(size=(3,) + n)
    v *= rng.uniform(0, 0.99, n) / np.sqrt((v * v).sum(0))
    v[:, rng.random(n) < 0.2] = 0.0
    nb = rng.uniform(0.1, 1.0, n)
    P = OR.params(shape, eos=eos)
    O = oracle()
    U = O.prim2cons(P, e, *v, nb)
    with S.Solver(shape, precision="fp64", eos="bag" if eos == OR.EOS_BAG else "ideal") as s:
        s.set_primitives(e, *v, nb)
        for a, b in zip(s.get_conserved(), U):
            assert max_rel_err(a, b) <= 1e-15
        got, ref = s.get_primitives(), O.recover(P, U)
        for k in ("e", "vx", "vy", "vz", "n", "p"):
            assert max_rel_err(got[k], ref[k]) <= 1e-13, k


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("name,slopes", [("ideal", [1 / 3]), ("kinked", [0.6, 0.0]), ("two values", [0.2])])
def test_table_primitives_against_extended_precision(name, slopes, precision):
    """The root M = (E + p(E - M v)) v of the tabulated EoS against a plain
    fixed point in extended precision: cells at rest, |v| from 1e-30 to 1 - 1e-9,
    energies below, in and above the table, and some (1e-25, 1e35) that leave
    the range of the float steps.  A last change of at most 1e-14 leaves
    1e-14 c / (1 - c) at a contraction c <= max p', and four roundings."""
    require_gpu()
    de, shape = 0.01, (50, 20, 4)
    nodes = 2 if name == "two values" else 1001
    table = np.concatenate([[0.0], np.cumsum(np.resize(slopes, nodes - 1) * de)])
    rng = np.random.default_rng(5)
    n = 4000
    E = 10.0 ** rng.uniform(-4, 2, n)
    frac = np.where(rng.random(n) < 0.5, rng.uniform(0, 1, n), 1 - 10.0 ** rng.uniform(-9, -1, n))
    frac[:200] = 10.0 ** rng.uniform(-30, -1, 200)
    frac[200:300] = 0.0
    if precision == "fp64":
        E[300:400], E[400:500] = 1e-25, 1e35
    M = E * frac
    if precision == "fp32":
        frac = np.minimum(frac, 1 - 1e-5)
        E = E.astype(np.float32).astype(np.float64)
        M = (E * frac).astype(np.float32).astype(np.float64)
    zero = np.zeros(n)
    with S.Solver(shape, precision=precision, check_input=False, autotune=False, eos="table", table=table,
                  table_de=de) as s:
        s.set_conserved([x.reshape(shape[::-1]) for x in (E, zero, M, zero, E)])
        got = s.get_primitives()
    T, h = table.astype(np.longdouble), np.longdouble(de)
    El, Ml = E.astype(np.longdouble), M.astype(np.longdouble)

    def p(e):
        k = np.clip(np.floor(e / h), 0, nodes - 2).astype(int)
        return T[k] + (e / h - k) * (T[k + 1] - T[k])

    v = Ml / (El + p(El))
    for _ in range(400):
        v = Ml / (El + p(El - Ml * v))
    c = max(slopes)
    tol = (1e-14 * c + 4 * 2.0 ** -52) / (1 - c)
    assert np.max(np.abs(got["vy"].ravel() - v)) <= tol
    assert np.max(np.abs(got["e"].ravel() - (El - Ml * v)) / El) <= tol
    assert np.max(np.abs(got["p"].ravel() - p(El - Ml * v)) / El) <= tol
    assert not got["vx"].any() and not got["vz"].any()
