"""Step-by-step parity of the CUDA path with the oracle (Alg. 1 steps).

Integer and index work is compared bit for bit (sparse-sign operator,
sparse-sign sketches, column exponents, pivots, breakdown indices); floating
point within tolerances derived from the arithmetic of each step.
"""
import numpy as np
import pytest
import scipy.linalg as sla
import torch

import oracle as O
import problems as P
from tests.gpu_util import dev_colmajor, to_np

pytestmark = pytest.mark.gpu

lsq = pytest.importorskip("paper_2603_16644_gb300")
U32 = 2.0 ** -24
U64 = 2.0 ** -53


@pytest.mark.parametrize("m,s,zeta,seed", [(1000, 200, 8, 5), (777, 31, 5, 3), (50, 8, 8, 1), (65536, 4096, 8, 2603),
                                           (3, 1, 1, 9)])
def test_sparse_sign_operator_bit_exact(m, s, zeta, seed):
    idx, sgn = lsq.sparse_sign_operator(seed, m, s, zeta)
    oi, os_ = O.sparse_sign_indices(seed, m, s, zeta)
    np.testing.assert_array_equal(to_np(idx), oi)
    np.testing.assert_array_equal(to_np(sgn), os_)


@pytest.mark.parametrize("prec", [O.FP8_E4M3, O.BF16, O.FP16, O.FP32, O.FP64])
def test_gaussian_operator(prec):
    """The ziggurat's proposals and its wedge test are IEEE products, sums and
    comparisons against the same tables, the grid rounding is exact: bit-exact.
    Only the tail (|z| > r, 0.026 % of the entries) goes through log, which
    differs by an ulp between libm and CUDA and can move an entry by one grid
    step (2^-17) next to a grid tie."""
    s, m, seed = 64, 3001, 77
    g = to_np(lsq.gaussian_operator(seed, s, m, prec))
    o = O.gaussian_operator(seed, s, m, prec)
    x, _ = O.zig_tables()
    tail = np.abs(O.gaussian_operator(seed, s, m, O.FP64)) > x[1]
    assert 10 < tail.sum() < 120, tail.sum()
    np.testing.assert_array_equal(g[~tail], o[~tail])
    gt, ot = g[tail], o[tail]
    neq = gt != ot
    assert neq.sum() <= 2
    if neq.any():
        p = {O.FP8_E4M3: 4, O.BF16: 8, O.FP16: 11, O.FP32: 24, O.FP64: 53}[prec]
        # a last-bit FP64 difference moves the grid value by one step, or
        # flips a rounding to the format, only next to a tie: neighbours
        step = np.maximum(2.0 ** -17, 2.0 ** (1 - p) * np.abs(ot[neq]))
        assert np.all(np.abs(gt[neq] - ot[neq]) <= 1.01 * step)


@pytest.mark.parametrize("prec", [O.FP8_E4M3, O.BF16, O.FP16, O.FP32, O.FP64])
@pytest.mark.parametrize("m,n,s,zeta", [(1037, 113, 300, 8), (2048, 64, 128, 4), (129, 65, 65, 3)])
def test_sparse_sketch_bit_exact(prec, m, n, s, zeta):
    rng = np.random.default_rng(m + n)
    A = np.asfortranarray(rng.standard_normal((m, n)) * np.exp2(rng.integers(-20, 20, n))[None, :])
    opts = lsq.make_opts(kind=lsq.SPARSE_SIGN, s=s, zeta=zeta, seed=42, sketch_prec=prec)
    As, ce, info = lsq.sketch(dev_colmajor(A), opts)
    oAs, oce = O.sketch(A, O.SPARSE_SIGN, s, zeta, 42, prec)
    assert int(to_np(info)[0]) == 0
    np.testing.assert_array_equal(to_np(ce), oce)
    np.testing.assert_array_equal(to_np(As).astype(np.float64), oAs)


def test_sparse_sketch_full_size_bit_exact():
    # the 65536 x 1024, s = 4096, zeta = 8, BF16 sketch of the tall-skinny workload
    m, n, s = 65536, 1024, 4096
    rng = np.random.default_rng(7)
    A = np.asfortranarray(rng.standard_normal((m, n)))
    opts = lsq.make_opts(kind=lsq.SPARSE_SIGN, s=s, zeta=8, seed=P.seed_for(1, 0), sketch_prec=lsq.BF16)
    As, ce, info = lsq.sketch(dev_colmajor(A), opts)
    oAs, oce = O.sketch(A, O.SPARSE_SIGN, s, 8, P.seed_for(1, 0), O.BF16)
    assert int(to_np(info)[0]) == 0
    np.testing.assert_array_equal(to_np(ce), oce)
    np.testing.assert_array_equal(to_np(As).astype(np.float64), oAs)


@pytest.mark.parametrize("prec", [O.FP8_E4M3, O.BF16, O.FP16, O.FP32, O.FP64])
@pytest.mark.parametrize("m,n,s", [(1037, 113, 300), (4096, 64, 192), (20011, 40, 120), (3, 2, 2)])
def test_srft_sketch_bit_exact(prec, m, n, s):
    # the butterflies of F are evaluated as in the oracle's sequential sweep
    # (levels in order, every pair the same sum and difference), the signs and
    # the sampled rows come from the same Philox words: bit for bit
    rng = np.random.default_rng(m + 3 * n)
    A = np.asfortranarray(rng.standard_normal((m, n)) * np.exp2(rng.integers(-20, 20, n))[None, :])
    opts = lsq.make_opts(kind=lsq.SRFT, s=s, zeta=0, seed=77, sketch_prec=prec)
    As, ce, info = lsq.sketch(dev_colmajor(A), opts)
    oAs, oce = O.sketch(A, O.SRFT, s, 0, 77, prec)
    assert int(to_np(info)[0]) == 0
    np.testing.assert_array_equal(to_np(ce), oce)
    np.testing.assert_array_equal(to_np(As).astype(np.float64), oAs)


@pytest.mark.parametrize("prec", [O.FP8_E4M3, O.FP32, O.FP64])
@pytest.mark.parametrize("m", [4, 17, 32, 33, 512, 513, 4095, 4097, 16384, 65537, 140000, 300000])
def test_srft_block_orders(prec, m):
    # orders below, at and above the 512 and 4096 entries that a warp and a CTA
    # hold, one to five and seven levels above: bit for bit, with entries that
    # round to subnormals and to zero, and a leading dimension above m
    n, s = 3, min(m, 70)
    rng = np.random.default_rng(m)
    A = np.asfortranarray(rng.standard_normal((m, n)) * np.exp2(rng.integers(-40, 1, (m, n))))
    A[rng.integers(0, m, 1 + m // 9), :] = 0.0
    A[m // 2, :] = [1.0, -3.0, 2.0**-30]
    opts = lsq.make_opts(kind=lsq.SRFT, s=s, zeta=0, seed=5, sketch_prec=prec)
    big = dev_colmajor(np.asfortranarray(np.vstack([A, np.full((3, n), np.nan)])))
    As, ce, info = lsq.sketch(big[:m], opts)
    oAs, oce = O.sketch(A, O.SRFT, s, 0, 5, prec)
    assert int(to_np(info)[0]) == 0
    np.testing.assert_array_equal(to_np(ce), oce)
    np.testing.assert_array_equal(to_np(As).astype(np.float64), oAs)


@pytest.mark.parametrize("prec", [O.FP8_E4M3, O.BF16, O.FP16, O.FP32, O.FP64])
def test_gaussian_sketch_within_rounding(prec):
    m, n, s = 1037, 113, 250
    rng = np.random.default_rng(3)
    A = np.asfortranarray(rng.standard_normal((m, n)))
    opts = lsq.make_opts(kind=lsq.GAUSSIAN, s=s, seed=9, sketch_prec=prec)
    As, ce, _ = lsq.sketch(dev_colmajor(A), opts)
    oAs, oce = O.sketch(A, O.GAUSSIAN, s, 0, 9, prec)
    np.testing.assert_array_equal(to_np(ce), oce)
    Om = O.gaussian_operator(9, s, m, prec)
    Ah = O.quantize(A, prec, oce)
    scale = np.abs(Om) @ np.abs(Ah)
    u = U64 if prec == O.FP64 else U32
    # both sums carry at most (m-1) u sum|terms|; operator entries may differ next to ties
    tol = 2 * m * u * scale + 2 ** -7 * np.abs(Ah).max() * 4
    if prec == O.FP64:
        # the FP64 sketch is a sum of K chunks of 1024 digit-sliced products,
        # each accurate to 1024 2^-50.6 2^3 max|A_chunk,c| (Omega sliced with
        # the fixed exponent 2^3 > |Omega|)
        dig = sum(1024 * 2.0 ** -50.6 * 8.0 * np.outer(np.ones(s), np.abs(Ah[k:k + 1024, :]).max(axis=0))
                  for k in range(0, m, 1024))
        tol = tol + dig
    assert np.all(np.abs(to_np(As) - oAs) <= tol)


@pytest.mark.parametrize("qr_prec", [O.FP32, O.FP64])
@pytest.mark.parametrize("s,n", [(300, 113), (256, 256), (4096, 200), (65, 1), (1000, 300), (1500, 600),
                                 (3000, 1030)])
def test_precond_qr(qr_prec, s, n):
    # FP64 with n > 256: blocks of 256 columns whose reflectors update the
    # later columns by digit-sliced tensor-core products (ragged last block)
    rng = np.random.default_rng(s + n)
    As = np.asfortranarray(rng.standard_normal((s, n)) @ np.diag(np.logspace(0, -2, n)))
    if qr_prec == O.FP32:
        As = O.round_to(As, O.FP32).reshape(As.shape, order="F")
    dt = torch.float32 if qr_prec == O.FP32 else torch.float64
    Ast = torch.from_numpy(np.ascontiguousarray(As.T)).cuda().to(dt).t()
    e = np.arange(n, dtype=np.int32) % 5 - 2
    R, info = lsq.precond_qr(Ast, torch.from_numpy(e).cuda(), qr_prec)
    R = to_np(R)
    assert int(to_np(info)[0]) == 0
    Ro = O.unscale_r(O.qr_r(As, qr_prec), e)
    assert np.all(np.diag(R) > 0) and np.all(np.tril(R, -1) == 0)
    u = U32 if qr_prec == O.FP32 else U64
    kap = O.kappa(As)
    # unique R with positive diagonal: both are backward-stable approximations of it
    Rc = np.linalg.cholesky(As.T @ As).T * np.exp2(-e)[None, :]
    dg = np.linalg.norm(R - Rc) / np.linalg.norm(Rc)
    do = np.linalg.norm(Ro - Rc) / np.linalg.norm(Rc)
    assert dg <= max(4 * do, 20 * n * u * kap), (dg, do)
    Ru = R * np.exp2(e)[None, :]
    assert np.linalg.norm(Ru.T @ Ru - As.T @ As) / np.linalg.norm(As) ** 2 <= 20 * s * u


@pytest.mark.parametrize("s,n", [(40, 33), (400, 64), (700, 40), (1900, 40), (2500, 40), (3500, 70), (5000, 70),
                                 (2100, 300)])
def test_precond_qr_fp64_rows_per_lane(s, n):
    """FP64 panels over every row count per lane (and more rows than the
    registers hold), columns graded over 2^+-60 and of either sign, against
    the oracle's R; both are columnwise backward stable, so every column of R
    is within a modest multiple of n u kappa of the other's, relative to the
    column (kappa of the matrix with its grading taken out)."""
    rng = np.random.default_rng(7 * s + n)
    B = rng.standard_normal((s, n))
    B[0] += 3.0 * np.where(np.arange(n) % 2, 1.0, -1.0)
    g = np.exp2(rng.integers(-60, 61, n))
    As = np.asfortranarray(B * g[None, :])
    R, info = lsq.precond_qr(dev_colmajor(As), None, O.FP64)
    R = to_np(R)
    assert int(to_np(info)[0]) == 0 and np.all(np.diag(R) > 0)
    Ro = O.qr_r(As, O.FP64)
    err = np.linalg.norm(R - Ro, axis=0) / np.linalg.norm(Ro, axis=0)
    assert err.max() <= 20 * n * U64 * O.kappa(B), err.max()


@pytest.mark.parametrize("s,n", [(64, 40), (65, 33), (128, 64), (129, 40), (257, 70), (513, 40), (1030, 33), (2500, 40),
                                 (4200, 40), (8192, 33), (8300, 40)])
def test_precond_qr_fp32_rows_and_clusters(s, n):
    """FP32 panels over every cluster size and row count per warp (and more rows
    than the registers hold): the bound of test_precond_qr_fp64_rows_per_lane
    with FP32's unit, columns graded over 2^+-30; and an upper triangular input
    comes back with its rows' signs made positive, exactly."""
    rng = np.random.default_rng(5 * s + n)
    B = rng.standard_normal((s, n))
    B[0] += 3.0 * np.where(np.arange(n) % 2, 1.0, -1.0)
    As = O.round_to(np.asfortranarray(B * np.exp2(rng.integers(-30, 31, n))[None, :]), O.FP32).reshape((s, n), order="F")

    def qr(M):
        R, info = lsq.precond_qr(torch.from_numpy(np.ascontiguousarray(M.T)).cuda().float().t(), None, O.FP32)
        assert int(to_np(info)[0]) == 0
        return to_np(R)

    R = qr(As)
    assert np.all(np.diag(R) > 0)
    Ro = np.linalg.qr(As, mode="r")
    Ro *= np.sign(np.diag(Ro))[:, None]
    err = np.linalg.norm(R - Ro, axis=0) / np.linalg.norm(Ro, axis=0)
    assert err.max() <= 20 * n * U32 * O.kappa(B), err.max()
    T = np.zeros((s, n))
    T[:n] = np.triu(As[:n])
    np.testing.assert_array_equal(qr(T), T[:n] * np.sign(np.diag(T))[:, None])


@pytest.mark.parametrize("s,n", [(200, 40), (1300, 70), (3000, 300)])
@pytest.mark.parametrize("prec,lo,hi", [(O.FP64, -516, -516), (O.FP64, -516, 0), (O.FP64, -500, 500), (O.FP64, 480, 480),
                                        (O.FP32, -64, -64), (O.FP32, -66, 63), (O.FP32, 60, 60)])
def test_precond_qr_extreme_column_norms(prec, lo, hi, s, n):
    """Columns with norms of 2^lo and 2^hi in turn, up to where their squares
    leave the normal range: finite, and columnwise within the bound of
    test_precond_qr_fp64_rows_per_lane, the unit enlarged by the rounding of a
    squared norm of s terms on the subnormal grid (2^-1074, FP32 2^-149)."""
    rng = np.random.default_rng(11 * s + n)
    B = rng.standard_normal((s, n))
    B[0] += 3.0 * np.sqrt(s) * np.where(np.arange(n) % 2, 1.0, -1.0)
    B /= np.linalg.norm(B, axis=0)
    e = np.where(np.arange(n) % 2, hi, lo).astype(float)
    As = B * np.exp2(e)
    u, grid = (U64, -1074) if prec == O.FP64 else (U32, -149)
    if prec == O.FP32:
        As = As.astype(np.float32).astype(np.float64)
    t = torch.from_numpy(np.ascontiguousarray(As.T)).cuda()
    R, info = lsq.precond_qr((t if prec == O.FP64 else t.float()).t(), None, prec)
    R = to_np(R)
    assert int(to_np(info)[0]) == 0 and np.isfinite(R).all() and np.all(np.diag(R) > 0)
    Bs = As * np.exp2(-e)
    Ro = np.linalg.qr(Bs, mode="r")
    Ro *= np.sign(np.diag(Ro))[:, None]
    err = np.linalg.norm(R * np.exp2(-e) - Ro, axis=0) / np.linalg.norm(Ro, axis=0)
    unit = u + s * 2.0 ** (grid - 2 * min(lo, hi))
    assert err.max() <= 20 * n * unit * O.kappa(Bs), err.max()


@pytest.mark.parametrize("s,n", [(513, 257), (1024, 300), (1025, 513), (1537, 600), (2600, 260)])
def test_precond_qr_fp64_block_products_over_chunks(s, n):
    """More than 256 columns: the block's products V^T [V C] over one to six
    chunks of 512 rows, the last one ragged, columns graded over 2^+-60: the bound
    of test_precond_qr_fp64_rows_per_lane, and R times a power of two exactly."""
    rng = np.random.default_rng(3 * s + n)
    B = rng.standard_normal((s, n))
    g = np.exp2(rng.integers(-60, 61, n))
    R, info = lsq.precond_qr(dev_colmajor(B * g), None, O.FP64)
    R = to_np(R)
    assert int(to_np(info)[0]) == 0
    Ro = np.linalg.qr(B, mode="r")
    Ro *= np.sign(np.diag(Ro))[:, None]
    err = np.linalg.norm(R / g - Ro, axis=0) / np.linalg.norm(Ro, axis=0)
    assert err.max() <= 20 * n * U64 * O.kappa(B), err.max()
    R2, _ = lsq.precond_qr(dev_colmajor(B * g * 2.0**-30), None, O.FP64)
    np.testing.assert_array_equal(to_np(R2), R * 2.0**-30)


def test_precond_qr_fp64_triangular_input():
    """Columns that are zero below the diagonal already (sigma = 0) with
    diagonal entries of either sign: R is the input with its rows' signs
    made positive, exactly, and a zero diagonal entry is a breakdown."""
    n = 45
    rng = np.random.default_rng(3)
    A = np.zeros((200, n))
    A[:n] = np.triu(rng.standard_normal((n, n)))
    R, info = lsq.precond_qr(dev_colmajor(A), None, O.FP64)
    assert int(to_np(info)[0]) == 0
    sg = np.sign(np.diag(A[:n]))
    np.testing.assert_array_equal(to_np(R), A[:n] * sg[:, None])
    A[20, 20] = 0.0
    _, info = lsq.precond_qr(dev_colmajor(A), None, O.FP64)
    assert int(to_np(info)[0]) == 21


def test_precond_qr_zero_column_reports_breakdown():
    s, n = 100, 10
    rng = np.random.default_rng(1)
    As = rng.standard_normal((s, n))
    As[:, 4] = 0.0
    Ast = torch.from_numpy(np.ascontiguousarray(As.T)).cuda().float().t()
    R, info = lsq.precond_qr(Ast, None, O.FP32)
    assert int(to_np(info)[0]) == 5


@pytest.mark.parametrize("hpne", [False, True])
@pytest.mark.parametrize("m,n,kap", [(1037, 113, 1e6), (3000, 200, 1e3), (500, 64, 1e8), (70, 1, 1.0)])
def test_trsm_gram(hpne, m, n, kap):
    pr = P.make_problem(m, n, kap, 1e-6, 1234)
    As, e = O.sketch(pr.A, O.SPARSE_SIGN, max(2 * n, 2), min(8, max(2 * n, 2)), 5, O.FP32)
    Rs = O.unscale_r(O.qr_r(As, O.FP32), e)
    Ap_o = O.trsm_right_upper(pr.A, Rs)
    G_o, c_o = O.gram(Ap_o, pr.A if hpne else Ap_o, pr.b)
    Ap, G, c = lsq.trsm_gram(dev_colmajor(pr.A), dev_colmajor(Rs), torch.from_numpy(pr.b).cuda(), hpne=hpne)
    Ap, G, c = to_np(Ap), to_np(G), to_np(c)
    kR = O.kappa(Rs)
    dAp = np.linalg.norm(Ap - Ap_o) / np.linalg.norm(Ap_o)
    assert dAp <= 4 * n * U64 * kR, dAp
    dG = np.linalg.norm(G - G_o) / np.linalg.norm(G_o)
    assert dG <= 2 * dAp * (np.linalg.norm(pr.A if hpne else Ap_o) * np.linalg.norm(Ap_o) / np.linalg.norm(G_o)) \
        + 4 * m * U64 * np.linalg.norm(Ap_o) ** 2 / np.linalg.norm(G_o), dG
    if not hpne:
        np.testing.assert_array_equal(G, G.T)
    dc = np.linalg.norm(c - c_o) / np.linalg.norm(c_o)
    assert dc <= 2 * dAp * np.linalg.norm(Ap_o) * np.linalg.norm(pr.b) / np.linalg.norm(c_o) + 4 * m * U64 * \
        np.linalg.norm(Ap_o) * np.linalg.norm(pr.b) / np.linalg.norm(c_o)


@pytest.mark.parametrize("n", [1, 7, 64, 65, 200, 1024, 1500])
def test_cholesky_solve(n):
    rng = np.random.default_rng(n)
    X = rng.standard_normal((3 * n + 5, n))
    G = X.T @ X
    c = rng.standard_normal(n)
    R = np.triu(rng.standard_normal((n, n))) + 5 * np.eye(n)
    L_o, info_o = O.cholesky(G)
    y_o = O.solve_upper(R, O.solve_lower_t(L_o, O.solve_lower(L_o, c)))
    x, F, _, info = lsq.factor_solve(dev_colmajor(G), torch.from_numpy(c).cuda(), Rs=dev_colmajor(R))
    assert int(to_np(info)[0]) == 0 == info_o
    kG = O.kappa(G)
    assert np.linalg.norm(to_np(F) - L_o) / np.linalg.norm(L_o) <= 8 * n * U64 * kG
    assert np.linalg.norm(to_np(x) - y_o) / np.linalg.norm(y_o) <= 8 * n * U64 * kG * O.kappa(R)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 127])
def test_cholesky_diagonal_block(n):
    """Orders around the 64-column block: against the oracle within the bound of
    test_cholesky_solve; a power of 4 in the matrix is the power of 2 in the
    factor, exactly, over the exponent range; every failing pivot is reported."""
    rng = np.random.default_rng(90 + n)
    X = rng.standard_normal((2 * n + 5, n))
    G = X.T @ X
    c = torch.zeros(n, dtype=torch.float64, device="cuda")
    L_o, _ = O.cholesky(G)
    F = to_np(lsq.factor_solve(dev_colmajor(G), c)[1])
    assert np.linalg.norm(F - L_o) / np.linalg.norm(L_o) <= 8 * n * U64 * O.kappa(G)
    for k in (-240, -17, 3, 250):
        Fk = to_np(lsq.factor_solve(dev_colmajor(G * 4.0**k), c)[1])
        np.testing.assert_array_equal(Fk, F * 2.0**k)
    for p in sorted({0, n // 3, n // 2, n - 1}):
        for v in (-1.0, np.inf):
            B = G.copy()
            B[p, p] = v
            assert int(to_np(lsq.factor_solve(dev_colmajor(B), c)[3])[0]) == O.cholesky(B)[1] == p + 1


@pytest.mark.parametrize("n", [130, 330, 449])
def test_cholesky_graded_pieces_componentwise(n):
    """Rows whose 64-column pieces of L are graded over 2^30 independently: the
    residual of every entry within (n + 1) u |L| |L|^T (the bound of Cholesky in
    FP64, for the FP64 operations) plus the digit products' 64 2^-50.6 times the
    two rows' largest entries, piece by piece, and a rounding of the entry."""
    rng = np.random.default_rng(60 + n)
    L0 = np.tril(rng.standard_normal((n, n)))
    L0 *= np.repeat(np.exp2(-rng.uniform(0, 30, (n, (n + 63) // 64))), 64, axis=1)[:, :n]
    L0[np.arange(n), np.arange(n)] = 2.0 * np.linalg.norm(np.tril(L0, -1), axis=1) + 2.0**-30
    G = L0 @ L0.T
    G = np.tril(G) + np.tril(G, -1).T
    x, F, _, info = lsq.factor_solve(dev_colmajor(G), torch.ones(n, dtype=torch.float64, device="cuda"))
    assert int(to_np(info)[0]) == 0
    F = np.tril(to_np(F))
    Fl = F.astype(np.longdouble)
    res = np.abs(Fl @ Fl.T - G).astype(np.float64)
    tol = (n + 1) * U64 * (np.abs(F) @ np.abs(F).T) + U64 * np.abs(G)
    for k in range(0, n, 64):
        mx = np.abs(F[:, k:k + 64]).max(axis=1)
        tol += 64 * 2.0**-50.6 * np.outer(mx, mx)
    assert np.all(res <= tol), (res / tol).max()


@pytest.mark.parametrize("n", [255, 256, 257, 320, 321, 577, 2100])
def test_cholesky_blocks(n):
    """Sizes around the 256-column blocks (inner updates of up to 192 columns,
    one product for the rest), against the oracle within the bound of
    test_cholesky_solve; the upper triangle is cleared, and a matrix that is
    not positive definite reports the pivot at which the oracle stops."""
    rng = np.random.default_rng(40 + n)
    X = rng.standard_normal((2 * n + 5, n))
    G = X.T @ X
    c = rng.standard_normal(n)
    L_o, info_o = O.cholesky(G)
    x, F, _, info = lsq.factor_solve(dev_colmajor(G), torch.from_numpy(c).cuda())
    F = to_np(F)
    assert int(to_np(info)[0]) == 0 == info_o and np.all(np.triu(F, 1) == 0)
    assert np.linalg.norm(F - L_o) / np.linalg.norm(L_o) <= 8 * n * U64 * O.kappa(G)
    k = n - 3
    G[k, k] = -1.0
    _, info_o = O.cholesky(G)
    _, _, _, info = lsq.factor_solve(dev_colmajor(G), torch.from_numpy(c).cuda())
    assert int(to_np(info)[0]) == info_o == k + 1


@pytest.mark.parametrize("n", [1, 5, 33, 64, 200, 1024])
def test_lu_solve(n):
    rng = np.random.default_rng(100 + n)
    H = rng.standard_normal((n, n)) + np.diag(np.full(n, 0.5))
    c = rng.standard_normal(n)
    LU_o, piv_o, info_o = O.lu(H)
    x_o = O.lu_solve(LU_o, piv_o, c)
    x, F, piv, info = lsq.factor_solve(dev_colmajor(H), torch.from_numpy(c).cuda(), hpne=True)
    assert int(to_np(info)[0]) == 0 == info_o
    np.testing.assert_array_equal(to_np(piv), piv_o)
    kH = O.kappa(H)
    assert np.linalg.norm(to_np(F) - LU_o) / np.linalg.norm(LU_o) <= 8 * n * U64 * kH
    assert np.linalg.norm(to_np(x) - x_o) / np.linalg.norm(x_o) <= 8 * n * U64 * kH


@pytest.mark.parametrize("n", [31, 32, 65, 129, 257, 520, 1030, 2100])
def test_lu_panel_rows_per_cluster(n):
    """The panel's cluster sizes (1 to 16 CTAs), rows per CTA and ragged last
    panels: the oracle's pivots, and factors within the bound of test_lu_solve;
    duplicate magnitudes in a column take the first largest pivot."""
    rng = np.random.default_rng(300 + n)
    H = rng.standard_normal((n, n)) + np.diag(np.full(n, 0.5))
    H[:, 0] = np.where(rng.random(n) < 0.5, -2.0, 2.0)  # ties in the first column
    c = rng.standard_normal(n)
    LU_o, piv_o, info_o = O.lu(H)
    x, F, piv, info = lsq.factor_solve(dev_colmajor(H), torch.from_numpy(c).cuda(), hpne=True)
    assert int(to_np(info)[0]) == 0 == info_o
    np.testing.assert_array_equal(to_np(piv), piv_o)
    kH = O.kappa(H)
    assert np.linalg.norm(to_np(F) - LU_o) / np.linalg.norm(LU_o) <= 8 * n * U64 * kH


@pytest.mark.parametrize("n", [30, 300, 700])
@pytest.mark.parametrize("d", [1.5, 3.0 * 2.0**1008, 1.3 * 2.0**-1000, 1.7 * 2.0**-1021, 5.0 * 2.0**-1074])
def test_lu_multipliers_are_the_divisions(n, d):
    """The first column's multipliers are entry / pivot as IEEE division gives
    them, bit for bit (the sign of zeros too), for entries over the whole
    exponent range below the pivot and for pivots down to subnormal ones."""
    rng = np.random.default_rng(n + int(np.log2(d)) + 2000)
    H = np.diag(np.full(n, 1.0)) + 0.01 * rng.standard_normal((n, n))
    col = d * rng.uniform(-1, 1, n) * np.exp2(-rng.uniform(0, 60, n))
    wide = rng.random(n) < 0.4
    col[wide] = (rng.uniform(-1, 1, n) * np.exp2(-rng.uniform(0, 1074, n)))[wide] * min(d, 1.0)
    col[rng.integers(0, n, 3)] = [0.0, -0.0, 2.0**-1074 if d > 2.0**-1070 else 0.0]
    at = int(rng.integers(0, n))
    col[at] = d
    H[:, 0] = col
    _, F, piv, _ = lsq.factor_solve(dev_colmajor(H), torch.ones(n, dtype=torch.float64, device="cuda"), hpne=True)
    F, piv = to_np(F), to_np(piv)
    assert piv[0] == at
    want = col.copy()
    for k in range(n):  # the row interchanges
        want[[k, piv[k]]] = want[[piv[k], k]]
    want[1:] = want[1:] / d
    np.testing.assert_array_equal(F[:, 0].view(np.int64), want.view(np.int64))


@pytest.mark.parametrize("n", [1, 40, 300])
def test_lu_zero_pivot_reported(n):
    """A zero column breaks down at its own index on both sides."""
    rng = np.random.default_rng(n)
    H = rng.standard_normal((n, n))
    H[:, n // 2] = 0.0
    _, _, info_o = O.lu(H)
    _, _, _, info = lsq.factor_solve(dev_colmajor(H), torch.ones(n, dtype=torch.float64).cuda(), hpne=True)
    assert int(to_np(info)[0]) == info_o == n // 2 + 1


def test_solve_wait_timeout_reports_and_recovers():
    """Fault injected on the host side (no GPU fault): with the test-only wait
    bound of the triangular solves cut to 1 ns, the blocks that find their
    predecessor's solution unpublished give up, record -2 in info and pass
    NaN on; the kernels return, and the next solve on the same context with
    the default bound is correct."""
    n = 1024
    rng = np.random.default_rng(11)
    X = rng.standard_normal((3 * n, n))
    G = X.T @ X
    c = rng.standard_normal(n)
    old = lsq.test_set_solve_wait_ns(1)
    try:
        _, _, _, info = lsq.factor_solve(dev_colmajor(G), torch.from_numpy(c).cuda())
        torch.cuda.synchronize()
        assert int(to_np(info)[0]) == -2
    finally:
        assert lsq.test_set_solve_wait_ns(old) == 1
    x, _, _, info = lsq.factor_solve(dev_colmajor(G), torch.from_numpy(c).cuda())
    assert int(to_np(info)[0]) == 0
    L_o, _ = O.cholesky(G)
    y_o = O.solve_lower_t(L_o, O.solve_lower(L_o, c))
    assert np.linalg.norm(to_np(x) - y_o) / np.linalg.norm(y_o) <= 8 * n * U64 * O.kappa(G)


def test_factor_breakdown_indices():
    G = np.diag([4.0, 1.0, -1.0, 2.0])
    _, _, _, info = lsq.factor_solve(dev_colmajor(G), torch.ones(4, dtype=torch.float64).cuda())
    assert int(to_np(info)[0]) == O.cholesky(G)[1] == 3
    H = np.array([[0.0, 1.0], [0.0, 2.0]])
    _, _, _, info = lsq.factor_solve(dev_colmajor(H), torch.ones(2, dtype=torch.float64).cuda(), hpne=True)
    assert int(to_np(info)[0]) == O.lu(H)[2] == 1


@pytest.mark.parametrize("kap", [1e1, 1e2, 1e3, 1e10])
def test_condest(kap):
    pr = P.make_problem(2000, 64, kap, 0.0, 91)
    k0, ch = lsq.condest(dev_colmajor(pr.A))
    k0, ch = float(to_np(k0)[0]), int(to_np(ch)[0])
    ok0, och, _, _, _ = O.condest(pr.A)
    if np.isinf(ok0):
        assert np.isinf(k0) and ch == och == O.FP64
    else:
        assert abs(k0 - ok0) <= 0.02, (k0, ok0)
        thresholds = np.array([2.0, 3.0, 4.0, 8.0])
        if np.min(np.abs(thresholds - ok0)) > 0.05:
            assert ch == och
