"""One step from a given tensor against the oracle over bond dimensions at the edges of the kernels' choices: every
compile-time bond dimension of the mode products and pair contractions, odd and uneven legs, one chunk and many chunks a
launch, one value of the outer axis and several; the eigensolver at every matrix size n = D^2 and at cluster sizes that
a batch sets; parity classes of unequal size.

Tolerances: an eigenvector of an n x n Gram matrix moves by n 2^-52 lambda_0 / gap under FP64 rounding (gap: the smallest
distance of a kept eigenvalue from its neighbours), and the tensor by as much for each of the up to six isometries; the
factor 8 covers the sums around them. The split-precision paths add FP32 rounding, 4 stages of at most 25 terms:
100 * 2^-24 = 6e-6, and the split's own 2^-16."""
import numpy as np
import pytest

from oracle import hotrg_ref as R
from tests.inputs import random_site_tensor, random_z2_site_tensor

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


def _flow(d, dcut, **kw):
    from paper_1906_06060_gb300 import HOTRG
    return HOTRG(d, 0.3, 0.0, dcut, **kw)


def _decaying(dims, seed):
    """Random tensor whose leg values weigh less from one to the next: separated Gram eigenvalues."""
    T = random_site_tensor(dims, seed=seed)
    for axis, n in enumerate(dims + dims):
        shape = [1] * (2 * len(dims))
        shape[axis] = n
        T = T * (0.8 ** np.arange(n)).reshape(shape)
    return T


def _tolerance(info):
    tol = 1e-13
    for iso in info.isometries.values():
        lam = iso.eigenvalues
        m = min(iso.chi, lam.size - 1)
        if m > 0:
            tol += 8 * lam.size * EPS * lam[0] / np.min(lam[:m] - lam[1:m + 1])
    return tol


def _check_step(dims, axis, dcut, extra=0.0, **kw):
    T = _decaying(dims, seed=sum(dims) + 31 * axis)
    ref, info = R.coarse_grain(T, axis, dcut)
    ref /= R.frobenius(ref)
    with _flow(len(dims), dcut, **kw) as f:
        f.set_tensor(T)
        f.step(axis)
        got = f.get_tensor()
        assert got.shape == ref.shape
        assert np.linalg.norm(got - ref) <= _tolerance(info) + extra
        for b, iso in info.isometries.items():
            np.testing.assert_allclose(f.spectra(1, b), iso.eigenvalues, rtol=0,
                                       atol=8 * iso.eigenvalues.size * EPS * iso.eigenvalues[0])


@pytest.mark.parametrize("dims,axis,dcut", [
    ((2, 3, 5, 4), 0, 5), ((5, 3, 2, 4), 1, 5), ((4, 4, 3, 3), 2, 4), ((3, 4, 4, 3), 3, 4), ((1, 2, 3, 2), 1, 4),
    ((6, 2, 3, 1), 2, 6),
    ((11, 4, 3), 2, 12), ((3, 13, 2), 0, 13), ((9, 5, 2), 1, 10), ((16, 2, 3), 2, 16), ((7, 6, 5), 0, 8),
    ((14, 2, 2), 1, 14), ((15, 2, 2), 2, 15), ((12, 3, 2), 1, 12)])
def test_fp64_step_matches_oracle(dims, axis, dcut):
    _check_step(dims, axis, dcut, precision="fp64")


@pytest.mark.parametrize("precision,extra", [("bf16x6", 1e-5), ("fp16x3", 1e-5), ("bf16x3", 4e-5)])
@pytest.mark.parametrize("dims,axis,dcut", [((4, 4, 4, 4), 3, 4), ((5, 4, 4, 5), 2, 5), ((5, 5, 3, 4), 0, 6),
                                            ((7, 9, 5), 1, 9)])
def test_split_precision_step_matches_oracle(precision, extra, dims, axis, dcut):
    _check_step(dims, axis, dcut, extra, precision=precision, fp64_steps=0)


@pytest.mark.parametrize("D", [2, 3, 4, 5, 7, 8, 9, 10, 11, 12, 13, 15, 16])
def test_eigensolver_sizes(D):
    """2D: one Gram matrix of D^2 rows, a cluster of its own."""
    _check_step((D, 3), 1, max(D, 3), precision="fp64")


@pytest.mark.parametrize("batch,D", [(3, 9), (20, 8), (40, 6), (160, 3)])
def test_eigensolver_clusters_of_a_batch(batch, D):
    """The matrices of a batch share the chip: fewer CTAs each. Every instance as alone, to FP64 rounding of its free
    energy over the steps of a short flow."""
    beta = np.linspace(0.40, 0.48, batch)
    from paper_1906_06060_gb300 import HOTRG
    with HOTRG(2, beta, 0.01, D, precision="fp64") as f:
        for _ in range(8):
            f.step()
        lnz = f.free_energy()[0]
    for i in (0, batch // 2, batch - 1):
        with HOTRG(2, float(beta[i]), 0.01, D, precision="fp64") as f:
            for _ in range(8):
                f.step()
            assert abs(f.free_energy()[0][0] - lnz[i]) < 1e-12


@pytest.mark.parametrize("dims,evens,axis", [((5, 4, 3, 4), (4, 1, 2, 3), 0), ((3, 5, 4, 5), (3, 1, 2, 2), 2),
                                             ((6, 2, 5), (1, 1, 4), 1), ((8, 8, 2), (7, 3, 1), 2)])
def test_uneven_parity_classes(dims, evens, axis):
    """Block-sparse and dense squeeze of one tensor: the norm and the spectra do not depend on the bonds' order. A 4D
    instance also runs the dense one over several outer values a launch, the block-sparse one over one."""
    T = random_z2_site_tensor(dims, evens, seed=5)
    out = []
    for z2 in (False, True):
        with _flow(len(dims), max(dims), z2=True, precision="fp64") as f:
            f.set_tensor(T, evens=evens if z2 else None)
            f.step(axis)
            out.append((f.ln_norms()[1], [f.spectra(1, b) for b in range(len(dims)) if b != axis]))
    assert abs(out[0][0] - out[1][0]) < 1e-12
    for a, b in zip(out[0][1], out[1][1]):
        np.testing.assert_allclose(b, a, rtol=0, atol=8 * a.size * EPS * a[0])


@pytest.mark.parametrize("precision", ["fp16x3", "bf16x6"])
@pytest.mark.parametrize("even", [0, 1, 2, 3, 4, 5, 8, 13])
def test_wide_parity_classes_in_split_precision(even, precision):
    """Classes of 0 to 13 values on the bond that the first zero-field contraction takes: the block-sparse against the dense
    squeeze of one tensor by what does not depend on the bonds' order, the norm and the next step's Gram spectra (FP32
    rounding, 6e-6, and the split's own 2^-16)."""
    dims, evens = (13, 5, 4), (even, 3, 2)
    T = random_z2_site_tensor(dims, evens, seed=even + 1)
    out = []
    for z2 in (False, True):
        with _flow(3, 13, z2=True, precision=precision, fp64_steps=0) as f:
            f.set_tensor(T, evens=evens if z2 else None)
            f.step(2)
            f.step(2)
            out.append((f.ln_norms()[1], [f.spectra(2, b) for b in (0, 1)]))
    assert abs(out[0][0] - out[1][0]) < 2.2e-5
    for a, b in zip(out[0][1], out[1][1]):
        np.testing.assert_allclose(b, a, rtol=0, atol=4.4e-5 * a[0])


@pytest.mark.parametrize("dims,axis,dcut", [((5, 4, 4, 4), 3, 5), ((4, 5, 4, 5), 3, 5), ((5, 5, 5, 4), 1, 5), ((2, 1), 1, 2),
                                            ((11, 11, 2), 2, 11)])
def test_gram_sums_over_a_few_columns_a_split(dims, axis, dcut):
    """Gram matrices over 2 to 12500 columns: four columns a split where there are not enough for the whole grid."""
    _check_step(dims, axis, dcut, precision="fp64")
