"""FP64 products by exact digit products: entries of very different size in one
block, digits at the end of their range, entries that are not finite.

An operand entry keeps its 53 bits down to 2^-17 of the largest one of its row
(column) and is rounded to 2^-71 of the row's power of two below that, so that
every element of a product is within a few roundings of 2^-53 of the sum of the
absolute values of its terms: what multiply-adds in FP64 give at best.
References: the operand itself (a product with the identity), and 64-bit-mantissa
sums of the exact inputs.
"""
import dataclasses
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@dataclasses.dataclass
class Sys:
    n_atoms: int
    pos: np.ndarray
    cell: None
    bsize: np.ndarray
    r_S: float
    r_H: float
    s_rowptr: np.ndarray
    s_col: np.ndarray
    s_val: np.ndarray
    h_rowptr: np.ndarray
    h_col: np.ndarray
    h_val: np.ndarray
    d_val: list


@pytest.fixture(scope="module")
def rt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1404_5776_gb300 as m
    m.build()
    return m


RADII = {k: 6.0 for k in ("r_Sinv", "r_T", "r_U", "r_K", "r_M")}


def _chain(H, b, spacing, S=None):
    """Atoms of b functions each on a line; the blocks of the dense H within 6 A, S diagonal (the identity by default)."""
    n = len(H) // b
    pos = np.zeros((n, 3))
    pos[:, 0] = spacing * np.arange(n)
    near = np.abs(pos[:, None, 0] - pos[None, :, 0]) < 6.0
    rowptr = np.concatenate([[0], np.cumsum(near.sum(1))]).astype(np.int32)
    blk = lambda M, i, j: M[i * b:(i + 1) * b, j * b:(j + 1) * b].reshape(-1)
    h = np.concatenate([blk(H, i, j) for i in range(n) for j in np.nonzero(near[i])[0]])
    S = np.eye(n * b) if S is None else S
    s = np.concatenate([blk(S, i, i) for i in range(n)])
    return Sys(n, pos, None, np.full(n, b, np.int32), 0.01, 6.0, np.arange(n + 1, dtype=np.int32),
               np.arange(n, dtype=np.int32), s, rowptr, np.nonzero(near)[1].astype(np.int32), h,
               [np.zeros_like(h)] * 3), near


def _dense(val, near, b):
    n = len(near)
    out, o = np.zeros((n * b, n * b), val.dtype), 0
    for i in range(n):
        for j in np.nonzero(near[i])[0]:
            out[i * b:(i + 1) * b, j * b:(j + 1) * b] = val[o:o + b * b].reshape(b, b)
            o += b * b
    return out


def _signs(rng, shape):
    return rng.choice([-1.0, 1.0], size=shape)


# 4-function systems of 20 atoms and more go in quads of four: with and without a last group of fewer
@pytest.mark.parametrize("b,n", [(13, 1), (13, 9), (4, 20), (4, 21), (4, 45)])
def test_product_with_the_identity_of_graded_entries(rt, b, n):
    rng = np.random.default_rng(b * n)
    N = b * n
    H = rng.uniform(0.5, 1.0, (N, N)) * _signs(rng, (N, N)) * 2.0 ** -rng.integers(0, 41, (N, N)).astype(float)
    H *= 2.0 ** rng.integers(-30, 31, N).astype(float)  # one scale per column
    s, near = _chain(H, b, 0.2)
    ctx = rt.RT(s, prop="em", dt=0.05, **RADII)
    ctx.inverse()
    ctx.propagator(0.0)
    T = _dense(ctx.matrix(0, rt.RT_MAT_T), near, b)  # S^-1 H with S = I
    ctx.close()
    H = H * np.kron(near, np.ones((b, b)))
    largest = np.abs(H).max(0)
    whole = np.abs(H) >= 2.0 ** -17 * largest
    assert np.array_equal(T.real[whole], H[whole]) and not T.imag.any()
    assert (np.abs(T.real - H) <= 2.0 ** -70 * largest).all()


def _square(rt, T, b, spacing):
    """cut(T T) from Re U = 1 - dt^2/2 cut(T T) of a three-term series with dt = 1, off its diagonal (0.5 is exact)."""
    s, near = _chain(T, b, spacing)
    ctx = rt.RT(s, prop="em", dt=1.0, taylor_terms=3, **RADII)
    ctx.inverse()
    ctx.propagator(0.0)
    U = _dense(ctx.matrix(0, rt.RT_MAT_U), near, b)
    ctx.close()
    off = np.kron(near, np.ones((b, b))).astype(bool) & ~np.eye(len(T), dtype=bool)
    return -2.0 * U.real, off


@pytest.mark.parametrize("grade", [0, 7, 14])
@pytest.mark.parametrize("b,n", [(13, 1), (13, 2), (13, 3), (13, 9), (4, 22), (4, 24), (4, 33)])
def test_every_element_of_a_graded_product(rt, b, n, grade):
    """T = D^-1 R D with D = 2^0..2^grade: the elements of T T span 2^+-grade, their terms one power of two each.
    A term is off by at most 2 2^(grade + 1) 2^-71 2^2 of itself (|R| in [0.5, 1)), at most 2^-53 for grade 14; the sum's one
    rounding is another 2^-53, and the digits left out stay below 2^-58."""
    rng = np.random.default_rng(100 * b + n + grade)
    N = b * n
    d = rng.integers(0, grade + 1, N).astype(float)
    T = rng.uniform(0.5, 1.0, (N, N)) * _signs(rng, (N, N)) * 2.0 ** (d[None, :] - d[:, None])
    got, off = _square(rt, T, b, 0.1)
    q = T.astype(np.longdouble)
    err = np.abs(got - q @ q).astype(float)
    assert (err <= 4.0 * 2.0 ** -53 * (np.abs(T) @ np.abs(T)))[off].all()


@pytest.mark.parametrize("b,n", [(13, 1), (13, 2), (13, 9), (13, 40), (4, 21), (4, 60)])
def test_sums_of_extreme_digits_are_exact(rt, b, n):
    """Every entry the same, its digits -64 and six times -256: the sums of a weight come as close to 2^24 between two
    carries as operands of 53 bits can bring them."""
    X = (1 << 69) + sum(256 << 9 * p for p in range(1, 7))
    x = -float(Fraction(X, 1 << 70))
    assert Fraction(-x) * (1 << 70) == X
    got, off = _square(rt, np.full((b * n, b * n), x), b, 0.1)
    exact = b * n * Fraction(x) ** 2
    assert len(set(got[off])) == 1
    assert abs(Fraction(got[off][0]) - exact) <= exact * Fraction(1, 1 << 53)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("b,n", [(13, 3), (4, 21)])
def test_entries_that_are_not_finite_stay_in_their_column(rt, b, n, bad):
    rng = np.random.default_rng(7)
    H = rng.uniform(0.5, 1.0, (b * n, b * n))
    H[1, b + 2] = bad
    s, near = _chain(H, b, 0.2)
    ctx = rt.RT(s, prop="em", dt=0.05, **RADII)
    ctx.inverse()
    ctx.propagator(0.0)
    T = _dense(ctx.matrix(0, rt.RT_MAT_T), near, b).real
    ctx.close()
    other = np.arange(b * n) != b + 2
    assert np.array_equal(T[:, other], H[:, other])
    assert not np.isfinite(T[:, b + 2]).any()  # 0 * inf and inf reach every row, as in multiply-adds


@pytest.mark.parametrize("cell,radius", [(3, 8.0), (4, 6.0)])
def test_product_of_two_propagators(rt, cell, radius):
    """ETRS without a field: U = cut(V V), V the EM propagator of half the step.  Every element within seven standard
    deviations of n roundings of |V||V| (2 sqrt(n) 2^-53), also where V falls by 2^20 among four neighbouring atoms."""
    import synth
    s = synth.diamond_system(cell, "sp4", 6.0, 6.0, seed=0)
    radii = {k: radius for k in RADII}
    got = []
    for prop, dt in (("etrs", 0.05), ("em", 0.025)):
        ctx = rt.RT(s, prop=prop, dt=dt, **radii)
        ctx.inverse()
        ctx.propagator(0.0)
        rowptr, col = ctx.pattern(0, rt.RT_PAT_U)
        near = np.zeros((s.n_atoms, s.n_atoms), bool)
        near[np.repeat(np.arange(s.n_atoms), np.diff(rowptr)), col] = True
        got.append(_dense(ctx.matrix(0, rt.RT_MAT_U), near, 4))
        ctx.close()
    U, V = got
    rows = np.arange(0, 4 * s.n_atoms, 37)
    cut = np.kron(near, np.ones((4, 4)))[rows]
    re, im = V.real.astype(np.longdouble), V.imag.astype(np.longdouble)
    exact_re, exact_im = re[rows] @ re - im[rows] @ im, re[rows] @ im + im[rows] @ re
    a, b = np.abs(V.real), np.abs(V.imag)
    n = 2 * 4 * near.sum(1).max()
    bound = 2.0 * np.sqrt(n) * 2.0 ** -53
    for part, exact, terms in ((U.real, exact_re, a[rows] @ a + b[rows] @ b), (U.imag, exact_im, a[rows] @ b + b[rows] @ a)):
        err = np.abs(part[rows] - exact * cut).astype(float)
        assert (err <= bound * terms * cut).all(), (err / np.where(terms > 0, terms, 1.0)).max()


@pytest.mark.parametrize("which,power", [(range(13), 0), (range(8, 13), 1), (range(8, 13), -1), (range(12, 13), -3), (range(0, 1), -2)])
def test_scaled_basis_functions(rt, which, power):
    """Some functions of every atom times 2^power, as far as the inverse's stopping rule goes along (2^2 up, 2^-5 down and
    it reports a stagnated residual): S^-1 H from the library's own S^-1, and one step's K' = U K U^dagger from its own U,
    every element within seven standard deviations of n roundings of the terms' absolute values."""
    import synth
    s = synth.diamond_system(2, "spd13", 7.0, 7.0, seed=0)
    n = 13 * s.n_atoms
    f = np.ones(13)
    f[list(which)] = 2.0 ** power
    outer = np.outer(f, f).reshape(-1)
    scale = lambda v: (v.reshape(-1, 169) * outer).reshape(-1)
    s = dataclasses.replace(s, s_val=scale(s.s_val), h_val=scale(s.h_val), d_val=[scale(d) for d in s.d_val])
    radii = {k: 8.0 for k in RADII}
    ctx = rt.RT(s, prop="em", dt=0.05, **radii)
    ctx.inverse()
    rowptr, col = ctx.pattern(0, rt.RT_PAT_U)
    near = np.zeros((s.n_atoms, s.n_atoms), bool)
    near[np.repeat(np.arange(s.n_atoms), np.diff(rowptr)), col] = True
    cut = np.kron(near, np.ones((13, 13))).astype(bool)
    rng = np.random.default_rng(1)
    K0 = rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n))
    K0 = (K0 + K0.conj().T) * cut / np.outer(np.tile(f, s.n_atoms), np.tile(f, s.n_atoms))
    ctx.set_density_dense(0, 0, K0)
    ctx.step(1)
    X, T, U, K = (_dense(ctx.matrix(0, m), near, 13) for m in (rt.RT_MAT_SINV, rt.RT_MAT_T, rt.RT_MAT_U, rt.RT_MAT_K))
    ctx.close()
    H, X, T = s.to_dense("H"), X.real, T.real
    rows = np.arange(0, n, 61)
    q = np.longdouble
    roundings = 2.0 * np.sqrt(n) * 2.0 ** -53
    err = np.abs(T[rows] - (X[rows].astype(q) @ H.astype(q)) * cut[rows]).astype(float)
    assert (err <= roundings * (np.abs(X[rows]) @ np.abs(H)) * cut[rows]).all()
    parts = lambda a: (a.real.astype(q), a.imag.astype(q))
    (ur, ui), (kr, ki), (vr, vi) = parts(U[rows]), parts(K0), parts(U)
    mr, mi = (ur @ kr - ui @ ki) * cut[rows], (ur @ ki + ui @ kr) * cut[rows]
    exact = (mr @ vr.T + mi @ vi.T) + 1j * (mi @ vr.T - mr @ vi.T)
    atom = np.arange(n) // 13
    up = cut[rows] & (atom[None, :] > atom[rows][:, None])
    terms = ((np.abs(U[rows]) @ np.abs(K0)) * cut[rows]) @ np.abs(U).T
    err = np.abs((K[rows] - exact).astype(complex))
    assert (err <= 4.0 * roundings * terms)[up].all()
