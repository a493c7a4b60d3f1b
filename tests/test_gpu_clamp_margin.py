"""The clamp |M| <= (1 - delta) E of the MIXED_FP64 recovery at margins where
the kernel's quick test of the high words has to hand over to the exact one.

Energies run over seven binades (their squares pass every significand) with
|M| / E up to 0.6% on both sides of 1 - delta.  The clamp count of a sweep is
that of a plain double evaluation of the float state, and the swept state that
of the oracle: some 30 float operations on values within a factor 2 of the
cell's energy give 30 * 2 * 2^-24 < 4e-6 of it (bound 1e-5), while one cell
that slips past the clamp moves its neighbours by 4e-5 to 4e-4 of it."""
import numpy as np
import pytest

from oracle import oracle as OR
from paper_1206_0919_gb300 import shasta as S
from gpu_util import oracle, require_gpu

pytestmark = pytest.mark.gpu

SHAPE = (96, 48, 10)


def state(delta, eos):
    nx, ny, nz = SHAPE
    rng = np.random.default_rng(int(1e6 * delta) + eos)
    x = np.arange(nx) / nx
    y = np.arange(ny) / ny
    E = 2.0 ** (3.5 + 3.5 * np.sin(2 * np.pi * (x[None, None, :] + y[None, :, None])))
    E = (E * np.ones((nz, 1, 1))).astype(np.float32).astype(np.float64)
    f = (1 - delta) * (1 + rng.uniform(-6e-3, 6e-3, E.shape))
    f = np.minimum(f, 1 - 1e-5)
    a = 0.5 + 0.4 * np.sin(2 * np.pi * y)[None, :, None]
    M = [(E * f * np.cos(a)), (E * f * np.sin(a) * 0.6), (E * f * np.sin(a) * 0.8)]
    M = [m.astype(np.float32).astype(np.float64) for m in M]
    M2 = M[0] ** 2 + M[1] ** 2 + M[2] ** 2
    lim = ((1 - delta) * E) ** 2
    near = np.abs(M2 / lim - 1) < 1e-12  # no rounding decides a cell
    for m in M:
        m[near] *= 0.5
    M2 = M[0] ** 2 + M[1] ** 2 + M[2] ** 2
    return [E, *M, E.copy()], int((M2 > lim).sum())


@pytest.mark.parametrize("tile", ["", "off"])
@pytest.mark.parametrize("eos", [OR.EOS_IDEAL, OR.EOS_BAG])
@pytest.mark.parametrize("delta", [0.005, 0.0075, 0.008, 0.0085, 0.009, 0.00999, 0.0101, 0.02])
def test_clamp_margin_against_double(monkeypatch, delta, eos, tile):
    require_gpu()
    monkeypatch.setenv("SHASTA_TILE", tile)
    U, over = state(delta, eos)
    assert 0 < over < U[0].size
    P = OR.params(SHAPE, bc=OR.BC_PERIODIC, eos=eos, delta=delta)
    for axis in range(3):
        with S.Solver(SHAPE, precision="mixed_fp64", bc="periodic", eos="bag" if eos else "ideal",
                      delta=delta, autotune=False) as s:
            s.set_conserved(U)
            s.sweep(axis)
            got, count = s.get_conserved(), s.counters()
        assert count == over, axis
        ref = oracle().sweep(P, U, axis)
        for g, r in zip(got, ref):
            assert np.max(np.abs(g - r) / U[0]) <= 1e-5, axis


@pytest.mark.parametrize("tile", ["", "off"])
@pytest.mark.parametrize("eos", [OR.EOS_IDEAL, OR.EOS_BAG])
@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e18])
def test_clamped_cells_against_oracle(monkeypatch, scale, eos, tile):
    """States of which most cells are clamped, |M| up to 3 E, at energies whose
    squares leave the range of float, against the oracle (the bound above, with
    |M| in the place of E); cells of E = 0 and E < 0 among them are counted."""
    require_gpu()
    monkeypatch.setenv("SHASTA_TILE", tile)
    nx, ny, nz = SHAPE
    U, _ = state(0.01, eos)
    x = np.arange(nx)[None, None, :] / nx
    U = [U[0] * scale] + [(m * scale * (1.7 + 1.3 * np.sin(4 * np.pi * x))) for m in U[1:4]] + [U[0].copy()]
    U = [u.astype(np.float32).astype(np.float64) for u in U]
    over = int((U[1] ** 2 + U[2] ** 2 + U[3] ** 2 > ((1 - 1e-6) * U[0]) ** 2).sum())
    assert over > U[0].size // 3
    P = OR.params(SHAPE, bc=OR.BC_PERIODIC, eos=eos, delta=1e-6)
    kw = dict(precision="mixed_fp64", bc="periodic", eos="bag" if eos else "ideal", check_input=False, autotune=False)
    with S.Solver(SHAPE, **kw) as s:
        for axis in range(3):
            s.set_conserved(U)
            s.sweep(axis)
            got = s.get_conserved()
            assert s.counters() == over, axis
            ref = oracle().sweep(P, U, axis)
            for k, (g, r) in enumerate(zip(got, ref)):
                assert np.max(np.abs(g - r) / (3 * U[0] / (scale if k == 4 else 1.0))) <= 1e-5, axis
        V = [u.copy() for u in U]
        V[0][:, ::7, 3::11] = 0.0
        V[0][:, 1::9, 5::13] *= -1.0
        M2 = V[1] ** 2 + V[2] ** 2 + V[3] ** 2
        bad = (V[0] <= 0) | (M2 > ((1 - 1e-6) * V[0]) ** 2)
        s.set_conserved(V)
        s.sweep(0)
        assert s.counters() == int(bad.sum())
