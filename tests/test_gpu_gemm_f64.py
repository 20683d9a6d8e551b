"""The FP64 product from exact integer slices (csrc/gemm_f64tc.cu) at the edges of its tiles, its ring and its sums."""
import math
from ctypes import c_void_p

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def gemm_f64(A, B, cta_group=1, pad=0):
    import torch
    from paper_1906_06060_gb300 import _lib
    lib = _lib.load()
    M, K = A.shape
    N = B.shape[0]
    a, b = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    C = torch.full((M, N + pad), -7.0, dtype=torch.float64, device="cuda")
    n = lib.hotrg_gemm_f64_scratch_bytes(M, N, K)
    scratch = torch.empty(n, dtype=torch.uint8, device="cuda")
    s = c_void_p(torch.cuda.current_stream().cuda_stream)
    _lib.check(lib.hotrg_gemm_f64(c_void_p(a.data_ptr()), K, c_void_p(b.data_ptr()), K, c_void_p(C.data_ptr()), N + pad,
                                  M, N, K, cta_group, c_void_p(scratch.data_ptr()), n, s), "hotrg_gemm_f64")
    _lib.check(lib.hotrg_gemm_status(c_void_p(scratch.data_ptr()), s), "status")
    out = C.cpu().numpy()
    assert np.all(out[:, N:] == -7.0)  # nothing beyond the columns is written
    return out[:, :N]


SHAPES = [(128, 256, 64), (129, 257, 65), (257, 511, 128), (256, 512, 1000), (300, 1030, 1023), (625, 260, 2049)]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("cta_group", [1, 2])
def test_integers_are_exact(M, N, K, cta_group):
    """Entries of at most 20 bits fit the rows' fixed-point numbers whatever their power-of-two scale, and their
    sums fit 53 bits: the product has no rounding at all."""
    rng = np.random.default_rng(M + N + K)
    a = rng.integers(-(2 ** 20) + 1, 2 ** 20, (M, K))
    b = rng.integers(-(2 ** 20) + 1, 2 ** 20, (N, K))
    a[3] = 0
    b[:, 0] = 2 ** 20 - 1
    ea, eb = rng.integers(-300, 300, M), rng.integers(-300, 300, N)
    ref = np.ldexp((a @ b.T).astype(np.float64), ea[:, None] + eb[None, :])
    got = gemm_f64(np.ldexp(a.astype(np.float64), ea[:, None]), np.ldexp(b.astype(np.float64), eb[:, None]), cta_group,
                   pad=(-N) % 4 + (4 if N % 2 else 0))
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("M,N,K", [(700, 20003, 64), (650, 16384, 200), (1100, 12289, 1090)])
@pytest.mark.parametrize("cta_group", [1, 2])
def test_several_tiles_of_a_cta_are_exact(M, N, K, cta_group):
    """More tiles than CTAs: a tile's results are formed between the next one's accumulator chains (few of them at one
    k-block), ragged tiles among them. Integers of 18 bits: no rounding."""
    rng = np.random.default_rng(K)
    a = rng.integers(-(2 ** 18), 2 ** 18, (M, K)).astype(np.float64)
    b = rng.integers(-(2 ** 18), 2 ** 18, (N, K)).astype(np.float64)
    assert np.array_equal(gemm_f64(a, b, cta_group, pad=(-N) % 4), a @ b.T)  # (sums below 2^53: exact in any order)


@pytest.mark.parametrize("signs", [False, True])
def test_largest_digits_fill_the_accumulators_exactly(signs):
    """Every digit at +-128, a whole number of accumulator chains: the sums reach their bounds. The exact value of an
    entry is an integer times (sum_i 2^(-8 i))^2, rounded once (and once more by the level-6 carry)."""
    from fractions import Fraction
    rng = np.random.default_rng(5)
    x = sum(2.0 ** (-8 * i) for i in range(7))  # the eighth digit does not fit a double beside the first
    M, N, K = 128, 256, 2048
    sa = np.where(rng.random((M, K)) < 0.5, -1.0, 1.0) if signs else np.ones((M, K))
    sb = np.where(rng.random((N, K)) < 0.5, -1.0, 1.0) if signs else np.ones((N, K))
    ref = (sa @ sb.T) * float(Fraction(x) ** 2)
    # fixed-point rows hold x exactly; far below one digit pair of the levels that are kept
    assert np.abs(gemm_f64(x * sa, x * sb) - ref).max() <= K * 2.0 ** -52


@pytest.mark.parametrize("M,N,K", [(300, 400, 777), (128, 300, 4100)])
@pytest.mark.parametrize("decay", [0.0, 0.01])
def test_error_is_below_the_fp64_chains(M, N, K, decay):
    """Gaussian rows, flat and decaying over many orders: against exactly summed products, within one rounding of the
    result plus K 2^-55 of the rows' largest entries (2^-56 from each operand's fixed point, entries of the other below
    its row's largest, and the dropped digit pairs), and in the 2-norm no further off than NumPy's FP64 product."""
    rng = np.random.default_rng(K)
    w = np.exp(-decay * np.arange(K))
    A, B = rng.standard_normal((M, K)) * w, rng.standard_normal((N, K)) * w
    got = gemm_f64(A, B)
    host = A @ B.T
    rows, cols = rng.integers(0, M, 300), rng.integers(0, N, 300)
    e, e_host = [], []
    for m, n in zip(rows, cols):
        p = A[m] * B[n]
        split = 134217729.0  # Dekker's exact product: p + err == A B
        ah, bh = A[m] * split, B[n] * split
        ah, bh = ah - (ah - A[m]), bh - (bh - B[n])
        al, bl = A[m] - ah, B[n] - bh
        err = ((ah * bh - p) + ah * bl + al * bh) + al * bl
        ref = math.fsum(np.concatenate([p, err]))
        tol = 2.0 ** -52 * abs(ref) + 2 * K * 2.0 ** -55 * np.abs(A[m]).max() * np.abs(B[n]).max()
        assert abs(got[m, n] - ref) <= tol
        e.append(got[m, n] - ref)
        e_host.append(host[m, n] - ref)
    assert np.linalg.norm(e) <= np.linalg.norm(e_host)


def test_non_finite_rows_and_zero_rows():
    rng = np.random.default_rng(0)
    A, B = rng.standard_normal((130, 100)), rng.standard_normal((300, 100))
    A[3, 5], A[7, 1], B[11, 99] = np.nan, np.inf, -np.inf
    A[20] = 0.0
    A[21] *= 1e-310  # subnormal entries
    C = gemm_f64(A, B)
    bad = np.zeros(C.shape, dtype=bool)
    bad[[3, 7]] = True
    bad[:, 11] = True
    assert np.array_equal(np.isnan(C), bad)
    assert np.all(C[20][~bad[20]] == 0.0)
    ref = A[21] @ np.where(np.isfinite(B), B, 0.0).T
    assert np.abs(C[21] - ref)[~bad[21]].max() <= 1e-320


@pytest.mark.parametrize("M,N,K", [(127, 256, 64), (128, 255, 64), (128, 256, 63), (128, 256, 16321)])
def test_shapes_it_does_not_take(M, N, K):
    from paper_1906_06060_gb300 import _lib
    lib = _lib.load()
    assert lib.hotrg_gemm_f64_scratch_bytes(M, N, K) == 0
    p = c_void_p(256)
    assert lib.hotrg_gemm_f64(p, K, p, K, p, N, M, N, K, 1, p, 1 << 40, None) == _lib.HOTRG_EINVAL


def _exact_dot(a, b):
    """Sum of a b, rounded once (Dekker's exact products)."""
    p, split = a * b, 134217729.0
    ah, bh = a * split, b * split
    ah, bh = ah - (ah - a), bh - (bh - b)
    al, bl = a - ah, b - bh
    return math.fsum(np.concatenate([p, ((ah * bh - p) + ah * bl + al * bh) + al * bl]))


@pytest.mark.parametrize("M,N,K,decay", [(300, 400, 600, 0.04), (130, 300, 128, 0.5), (257, 260, 2049, 0.02),
                                         (128, 256, 64, -0.9)])
@pytest.mark.parametrize("cta_group", [1, 2])
def test_columns_that_grow_where_the_others_decay(M, N, K, decay, cta_group):
    """A decays along k as Bt grows, by up to 28 orders: the products are of one size, and what counts are each row's
    small entries. Error: a rounding and (2^-53 + K 2^-58) of the product of the rows' largest entries after the
    power-of-two column scales (the sizes of Bt's columns); in the 2-norm no further off than NumPy's FP64 product."""
    rng = np.random.default_rng(K)
    A = rng.standard_normal((M, K)) * np.exp(-decay * np.arange(K))
    B = rng.standard_normal((N, K)) * np.exp(decay * np.arange(K))
    got = gemm_f64(A, B, cta_group)
    host = A @ B.T
    c = np.ldexp(1.0, np.frexp(np.abs(B).max(0))[1] - 1)
    ra, rb = np.abs(A * c).max(1), np.abs(B / c).max(1)
    e, e_host = [], []
    for m, n in zip(rng.integers(0, M, 300), rng.integers(0, N, 300)):
        ref = _exact_dot(A[m], B[n])
        assert abs(got[m, n] - ref) <= 2.0 ** -53 * abs(ref) + (2.0 ** -53 + K * 2.0 ** -58) * ra[m] * rb[n]
        e.append(got[m, n] - ref)
        e_host.append(host[m, n] - ref)
    assert np.linalg.norm(e) <= np.linalg.norm(e_host)


def test_columns_of_zeros_and_extreme_columns():
    """A column of zeros of Bt leaves no trace of A's entries there, however large, unless they are not finite; columns at
    the ends of the exponent range, subnormal ones included, cancel in the scales. Integers: no rounding."""
    rng = np.random.default_rng(1)
    M, N, K = 130, 300, 100
    a = rng.integers(-(2 ** 20) + 1, 2 ** 20, (M, K))
    b = rng.integers(-(2 ** 20) + 1, 2 ** 20, (N, K))
    b[:, 7] = 0
    ref = (a @ b.T).astype(np.float64)
    g = rng.integers(-900, 900, K)
    g[[3, 4]] = 1000, -1000
    A, B = np.ldexp(a.astype(np.float64), -g), np.ldexp(b.astype(np.float64), g)
    A[:, 7] = 1e300
    B[:, 11] = np.ldexp(b[:, 11].astype(np.float64), -1074)
    A[:, 11] = np.ldexp(a[:, 11].astype(np.float64), 1000)
    ref = (ref - np.outer(a[:, 11], b[:, 11])) + np.ldexp(np.outer(a[:, 11], b[:, 11]).astype(np.float64), -74)
    A[9, 7] = np.nan
    got = gemm_f64(A, B)
    assert np.all(np.isnan(got[9]))
    keep = np.arange(M) != 9
    # (column 11 is 2^-74 of the others: the sum of the two rounds once)
    assert np.abs(got - ref)[keep].max() <= 2.0 ** -52 * np.abs(ref).max()


def test_step_of_a_tensor_in_an_unbalanced_gauge():
    """The bond along the merged axis scaled by 2^-12 i on its lower leg and 2^12 i on its upper one: the same contraction,
    from operands whose rows spread over 36 bits in opposite directions. Every block of the new tensor (a pair of values of
    the outer legs of that axis) against the oracle, to the rounding that the isometries allow: 8 n eps lambda_0 / gap for
    each of six, as a step from a balanced tensor, and 1e-13."""
    from oracle import hotrg_ref as R
    from paper_1906_06060_gb300 import HOTRG
    from tests.inputs import random_site_tensor
    n = 4
    T = random_site_tensor((n,) * 4, seed=3)
    for axis in range(8):
        shape = [1] * 8
        shape[axis] = n
        T = T * (0.8 ** np.arange(n)).reshape(shape)
    g = np.ldexp(1.0, 12 * np.arange(n))
    T = T / g.reshape((1, 1, 1, n, 1, 1, 1, 1)) * g
    ref, info = R.coarse_grain(T, 3, n)
    ref /= R.frobenius(ref)
    tol = 1e-13
    for iso in info.isometries.values():
        lam = iso.eigenvalues
        tol += 8 * lam.size * 2.0 ** -52 * lam[0] / np.min(lam[:n] - lam[1:n + 1])
    with HOTRG(4, 0.3, 0.0, n, precision="fp64") as f:
        f.set_tensor(T)
        f.step(3)
        got = f.get_tensor()
    for u in range(n):
        for p in range(n):
            x, y = got[:, :, :, u, :, :, :, p], ref[:, :, :, u, :, :, :, p]
            assert np.linalg.norm(x - y) <= tol * np.linalg.norm(y), (u, p)


def test_waits_that_run_out_leave_the_device_usable():
    """The wait probe's FP64 launches (one CTA; pairs whose CTAs issue no copies, or only one of them does) give up within
    their limit, and exact products follow on the same device."""
    import time

    import torch
    from paper_1906_06060_gb300 import _lib
    lib = _lib.load()
    n = lib.hotrg_gemm_wait_probe_bytes()
    scratch = torch.zeros(n, dtype=torch.uint8, device="cuda")
    s = c_void_p(torch.cuda.current_stream().cuda_stream)
    t0 = time.time()
    for _ in range(3):
        assert lib.hotrg_gemm_wait_probe(0.05, c_void_p(scratch.data_ptr()), n, s) == _lib.HOTRG_ETIMEOUT
    assert time.time() - t0 < 10.0  # six launches of one limit each, a drain of a second at most in each
    rng = np.random.default_rng(2)
    a, b = rng.integers(-1000, 1000, (300, 200)).astype(np.float64), rng.integers(-1000, 1000, (520, 200)).astype(np.float64)
    for cta_group in (1, 2):
        assert np.array_equal(gemm_f64(a, b, cta_group), a @ b.T)


def _cut(x, column_exponents):
    """The kernel's digits of one row (entry k scaled by 2^column_exponents[k] first) and the row's exponent."""
    man, ex = np.frexp(x)
    man = np.ldexp(man, 53).astype(np.int64)
    ex = ex + column_exponents
    e = int(ex[x != 0].max())
    shift = ex - e + 10  # x 2^(63 - e) = man 2^shift
    v = np.where(shift >= 0, man << np.clip(shift, 0, 10),
                 np.sign(man) * ((np.abs(man) + (np.int64(1) << np.clip(-shift - 1, 0, 60))) >> np.clip(-shift, 0, 61)))
    digits = np.zeros((8, x.size), dtype=np.int64)
    for i in range(7, 0, -1):
        digits[i] = ((v & 255) ^ 128) - 128
        v = (v - digits[i]) >> 8
    digits[0] = v
    return digits, e


@pytest.mark.parametrize("M,N,K,cta_group", [(128, 256, 1024, 1), (128, 256, 16320, 1), (300, 256, 16320, 2),
                                             (130, 257, 16319, 2)])
def test_extreme_digits_are_summed_exactly(M, N, K, cta_group):
    """Rows whose digits are all at the ends of their range: accumulator chains up to 15/16 of 2^24, level sums up to 7/8
    of 2^31, carries between levels of that size. The kernel's arithmetic in Python's integers, rounded once, gives the
    same bits."""
    from fractions import Fraction
    rng = np.random.default_rng(K)
    low = np.ldexp(float(-0x7F80808080808000), -63)    # digits -127, -128 (six times), 0
    high = np.ldexp(float(0x7F7F7F7F7F7F7C00), -63)    # 127 (six times), 124, 0
    tail = np.ldexp(float(-0x80808080808080), -63)     # 0, -128 (seven times)
    rows = np.array([np.full(K, low), np.full(K, high), np.where(np.arange(K) % 2, low, -low),
                     np.concatenate([[high], np.full(K - 1, tail)]), rng.choice([low, -low, high, -high, tail, -tail], K)])
    c = np.frexp(np.abs(rows).max(0))[1] - 1
    a = [_cut(x, c) for x in rows]
    b = [_cut(x, -c) for x in rows]
    assert a[0][0][:, 5].tolist() == [-127] + [-128] * 6 + [0] and a[1][0][:, 5].tolist() == [127] * 6 + [124, 0]
    assert a[3][0][:, 5].tolist() == [0] + [-128] * 7
    ref, largest = np.zeros((5, 5)), 0
    for i, (qa, ea) in enumerate(a):
        for j, (qb, eb) in enumerate(b):
            level = [sum(int(qa[u] @ qb[s - u]) for u in range(s + 1)) for s in range(8)]
            largest = max(largest, max(abs(x) for x in level))
            level[6] += (level[7] + 128) >> 8
            level[5] += (level[6] + 128) >> 8
            assert max(abs(x) for x in level) < 2 ** 31 - 128
            ref[i, j] = float(sum(Fraction(level[s], 2 ** (14 + 8 * s)) for s in range(6)) * Fraction(2) ** (ea + eb))
    assert largest > 6.9 * 2 ** 14 * K  # seven pairs of (nearly) extreme digits
    got = gemm_f64(rows[np.arange(M) % 5], rows[np.arange(N) % 5], cta_group)
    assert np.array_equal(got, ref[np.arange(M) % 5][:, np.arange(N) % 5])
