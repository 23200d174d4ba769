"""FP64 products by exact digit products (tensor cores): 13-function blocks, and
4-function blocks in quads of four consecutive atoms.

The digits are exact, so a product with the identity has to return the other
operand bit for bit wherever its entries keep 53 bits above the last digit
(2^-70 of the column's scale: entries from 2^-16 of its maximum on), the others
to within that digit, whatever the scales of its columns; and a Taylor series of random blocks has to
agree with dense 64-bit algebra within the rounding of the latter.  Sizes: one
atom, fewer and more triples than one carry interval (8), block sizes below 13
(padding), blocks that leave leading digits at zero.
"""
import dataclasses

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


def _chain(n, bsize, block, r=6.0, spacing=1.0):
    """Atoms on a line, S = I, H_ij = block(i, j) within r."""
    pos = np.zeros((n, 3))
    pos[:, 0] = spacing * np.arange(n)
    near = np.abs(pos[:, None, 0] - pos[None, :, 0]) < r
    rowptr = np.concatenate([[0], np.cumsum(near.sum(1))]).astype(np.int32)
    col = np.nonzero(near)[1].astype(np.int32)
    h = np.concatenate([block(i, j).reshape(-1) for i in range(n) for j in np.nonzero(near[i])[0]])
    eye = np.concatenate([np.eye(b).reshape(-1) for b in bsize])
    return Sys(n, pos, None, np.asarray(bsize, np.int32), 0.5, r, np.arange(n + 1, dtype=np.int32),
               np.arange(n, dtype=np.int32), eye, rowptr, col, h, [np.zeros_like(h)] * 3), near


def _dense(s, near, val):
    off = np.concatenate([[0], np.cumsum(s.bsize)])
    out, o = np.zeros((off[-1], off[-1]), val.dtype), 0
    for i in range(s.n_atoms):
        for j in np.nonzero(near[i])[0]:
            k = s.bsize[i] * s.bsize[j]
            out[off[i]:off[i + 1], off[j]:off[j + 1]] = val[o:o + k].reshape(s.bsize[i], s.bsize[j])
            o += k
    return out


@pytest.mark.parametrize("n,bsize", [(1, [13]), (2, [13, 1]), (9, [13, 12, 5, 13, 13, 9, 13, 4, 13]), (40, [13] * 40)])
@pytest.mark.parametrize("spread", [0, 30, 200])
def test_product_with_the_identity_is_exact(rt, n, bsize, spread):
    rng = np.random.default_rng(n + spread)
    expo = [rng.integers(-spread, spread + 1, size=b) for b in bsize]  # one scale per column of H

    def block(i, j):
        m = rng.uniform(0.5, 1.0, size=(bsize[i], bsize[j])) * rng.choice([-1.0, 1.0], size=(bsize[i], bsize[j]))
        far = 2.0 ** (-9.0 * abs(i - j))  # leading digits of far blocks are zero
        return m * far * 2.0 ** expo[j][None, :].astype(float)

    s, near = _chain(n, bsize, block)
    ctx = rt.RT(s, prop="em", dt=0.05, **{k: 6.0 for k in ("r_Sinv", "r_T", "r_U", "r_K", "r_M")})
    ctx.inverse()
    ctx.propagator(0.0)
    T = ctx.matrix(0, rt.RT_MAT_T)  # S^-1 H with S^-1 = I
    ctx.close()
    T, H = _dense(s, near, T), _dense(s, near, s.h_val)
    largest = np.abs(H).max(0)
    whole = np.abs(H) >= 2.0 ** -16 * largest
    assert np.array_equal(T.real[whole], H[whole]) and not T.imag.any()
    assert (np.abs(T.real - H) <= 2.0 ** -69 * largest).all()


@pytest.mark.parametrize("most", [13, 4])
@pytest.mark.parametrize("n,spacing", [(1, 1.0), (3, 1.0), (9, 1.0), (20, 0.5), (70, 0.1)])
def test_series_and_sandwich_against_dense_algebra(rt, n, spacing, most):
    """U and K' = U K U^dagger from random decaying blocks (1 to 70 triples an item; r = 6; 4-function
    systems with and without a last group of fewer than four atoms)."""
    rng = np.random.default_rng(n)
    bsize = rng.integers(1, most + 1, size=n)
    bsize[0] = most
    raw = {}

    def block(i, j):
        if (j, i) in raw:
            return raw[j, i].T
        raw[i, j] = rng.normal(size=(bsize[i], bsize[j])) * np.exp(-2.0 * abs(i - j) * spacing)
        if i == j:
            raw[i, j] = raw[i, j] + raw[i, j].T
        return raw[i, j]

    s, near = _chain(n, bsize, block, spacing=spacing)
    radii = {k: 6.0 for k in ("r_Sinv", "r_T", "r_U", "r_K", "r_M")}
    ctx = rt.RT(s, prop="em", dt=0.05, **radii)
    ctx.inverse()
    K0 = rng.normal(size=(bsize.sum(),) * 2) + 1j * rng.normal(size=(bsize.sum(),) * 2)
    mask = np.repeat(np.repeat(near, bsize, 0), bsize, 1)
    K0 = (K0 + K0.conj().T) * mask
    ctx.set_density_dense(0, 0, K0)
    ctx.step(1)
    U, K = _dense(s, near, ctx.matrix(0, rt.RT_MAT_U)), _dense(s, near, ctx.matrix(0, rt.RT_MAT_K))
    ctx.close()
    T = _dense(s, near, s.h_val)
    ref, P, c = np.eye(len(T)) - 0.05j * T, T, -0.05j
    for m in range(2, 6):
        P = (T @ P) * mask
        c = c * -0.05j / m
        ref = ref + c * P
    Kref = (((ref @ K0) * mask) @ ref.conj().T) * mask
    # with M cut K' is not hermitian by itself: the upper blocks are mirrored, the diagonal ones symmetrised
    atom = np.repeat(np.arange(n), bsize)
    up, on = atom[:, None] < atom[None, :], atom[:, None] == atom[None, :]
    Kref = Kref * up + (Kref * up).conj().T + 0.5 * (Kref + Kref.conj().T) * on
    # rounding of N-term 64-bit sums in the reference: N 2^-53 of row norm x column norm, per product
    N, eps = len(T), 2.0 ** -53
    norm = lambda A: np.linalg.norm(A, axis=1).max()
    series = sum((0.05 * norm(T)) ** m for m in range(6))
    assert np.abs(U - ref).max() <= 6 * N * eps * series
    assert np.abs(K - Kref).max() <= 4 * N * eps * series ** 2 * norm(K0)
