"""Rotation angles of the Jacobi eigensolver: a block of small entries beside a large one.

The tensor's Gram matrix is 1 at one index and holds two 2 x 2 blocks of entries near s^2 = 2^-34, everything else zero
but products of two such blocks (2^-68). Its entries are exact in FP64 and the large entry couples to nothing, so each
block's eigenvectors are known from one rotation. The blocks' entries (1e-10) lie far above the rotation threshold
(2^-53 of the norm), 1e-7 of them far below it: what a single-precision angle leaves is never rotated again and would
stay in the vectors (6e-8); the solver corrects the angle to about the product of two such errors (1e-14)."""
import numpy as np
import pytest

from oracle import hotrg_ref as R

pytestmark = pytest.mark.gpu

S = 2.0 ** -17


def _tensor(D, x, p, q, m1, m2):
    """T[u0, u1, p0, p1] of bond dimensions (D, 2) whose Gram matrix along axis 1 is (A A^T + B B^T) x (A A^T) with
    A = 1 at (x, x) and S m1 at (p, q), B = S m2 at (p, q)."""
    A, B = np.zeros((D, D)), np.zeros((D, D))
    A[x, x] = 1.0
    A[np.ix_((p, q), (p, q))] = S * m1
    B[np.ix_((p, q), (p, q))] = S * m2
    T = np.zeros((D, 2, D, 2))
    T[:, 0, :, 0] = A
    T[:, 1, :, 0] = B
    return T


def _vectors(a):
    """Eigenvalues and vectors (columns) of a symmetric 2 x 2 matrix, the larger component positive."""
    t = 0.5 * np.arctan2(2 * a[0, 1], a[0, 0] - a[1, 1])
    v = np.array([[np.cos(t), -np.sin(t)], [np.sin(t), np.cos(t)]])
    v *= np.sign(v[np.abs(v).argmax(0), np.arange(2)])
    c, s = np.cos(t), np.sin(t)
    cross = 2 * c * s * a[0, 1]
    return np.array([c * c * a[0, 0] + s * s * a[1, 1] + cross, s * s * a[0, 0] + c * c * a[1, 1] - cross]), v


@pytest.mark.parametrize("D,x,p,q", [(3, 0, 1, 2), (4, 2, 0, 3), (8, 5, 1, 6), (9, 0, 3, 7), (13, 12, 4, 5), (16, 7, 0, 15)])
def test_vectors_of_a_small_block(D, x, p, q):
    """n = D^2 = 9 to 256, both forms of the rotation. A corrected angle is off by at most 3e-14 (the correction's own
    single-precision error, 3 roundings of 2^-24 on 1.5e-7), the new tensor's entries of two such vectors by 6e-14 of
    S |m|, and FP64 rounding adds less than 4e-14: 1e-13 in all."""
    from paper_1906_06060_gb300 import HOTRG
    rng = np.random.default_rng(D)
    for _ in range(12):
        while True:  # eigenvalues apart from one another, vectors with no tie of components
            m1, m2 = rng.integers(-4, 5, (2, 2)).astype(float), rng.integers(-4, 5, (2, 2)).astype(float)
            S2 = m1 @ m1.T
            S1 = S2 + m2 @ m2.T
            (l1, v1), (l2, v2) = _vectors(S1), _vectors(S2)
            lam = np.concatenate([l1, l2])
            near = min(abs(abs(v[0, k]) - abs(v[1, k])) for v in (v1, v2) for k in (0, 1))
            if S1[0, 1] and S2[0, 1] and np.diff(np.sort(np.append(lam, 0.0))).min() > 0.2 and near > 0.05:
                break
        T = _tensor(D, x, p, q, m1, m2)
        U = np.zeros((D, D, 5))
        U[x, x, 0] = 1.0
        for k, o in enumerate(np.argsort(-lam)):
            if o < 2:
                U[(p, q), (x, x), k + 1] = v1[:, o]
            else:
                U[(x, x), (p, q), k + 1] = v2[:, o - 2]
        ref = R.squeeze(T, T, 1, {0: U})
        ref /= R.frobenius(ref)
        with HOTRG(2, 0.3, 0.0, max(D, 5), precision="fp64") as f:
            f.set_tensor(T)
            f.step(1)
            got = f.get_tensor()[:5, :, :5, :]
        scale = np.abs(np.concatenate([m1, m2])).max()
        assert np.abs(got - ref)[1:, :, 1:, :].max() <= 1e-13 * S * scale
        assert np.abs(got - ref).max() <= 1e-13
