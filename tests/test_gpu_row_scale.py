"""Row-wise accuracy of the FP64 path on matrices whose rows differ in scale.

Householder QR is backward stable row by row where the heavy rows come first (Cox and
Higham, BIT 38, 1998): A + dA = Q R with |dA_ij| <= c u alpha_i, alpha_i the largest
magnitude row i has during the factorization, however far the rows' scales are apart.
The factor c holds the growth of the light rows, which is the matrix's; it is taken from
the sequential oracle on the same matrix.  The checks form A - Q R, or apply the stored
reflectors, in extended precision, and compare row by row.

Bound: blocked sums round in another order than the oracle's, and the largest of m n
such errors scatters, so the GPU may have 8 times the oracle's largest row error, plus
4 sqrt(n) u alpha_i (n updates of a few u alpha_i each, as a random walk).  There is no
weight in it.
"""
import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_fp64_tc import ctx  # noqa: F401
from test_gpu_parity import U, dev, host

pytestmark = pytest.mark.gpu

WEIGHTS = [1.0, 2.0 ** 9, 2.0 ** 13, 2.0 ** 33, 2.0 ** 60]


def apply_q(F, up, X, transpose=False):
    """Q X (or Q^T X) in extended precision, reflector by reflector."""
    F, X = F.astype(np.longdouble), X.astype(np.longdouble)
    n = min(F.shape[1], F.shape[0] - 1)
    for k in (range(n) if transpose else reversed(range(n))):
        if up[k] == 0.0:
            continue
        v = F[k:, k].copy()
        v[0] = up[k]
        b = v[0] * F[k, k]
        X[k:] += np.outer(v, (v @ X[k:]) / b)
    return X


def row_errors(A, F, up):
    """max_j |A - Q R|_ij / alpha_i."""
    n = A.shape[1]
    R = np.zeros_like(A)
    R[:n] = np.triu(F[:n])
    E = np.abs(A - apply_q(F, up, R)).max(axis=1)
    alpha = np.abs(A).max(axis=1)
    alpha[:n] = np.maximum(alpha[:n], np.abs(R[:n]).max(axis=1))
    return (E / alpha).astype(float)


def bound(eo, n):
    return 8.0 * eo + 4.0 * np.sqrt(n) * U


def report(label, w, eo, eg, n):
    print(f"ROWERR {label} w=2^{np.log2(w):.0f} oracle {eo / U:.1f}u gpu {eg / U:.1f}u")
    assert eg <= bound(eo, n)


def heavy_top(m, n, h, w, seed):
    A, _ = workloads.gaussian(m, n, seed=seed)
    A = np.array(A)
    A[:h] *= w
    return A


LIGHT = 96       # columns the heavy rows of block_sparse do not touch


def block_sparse(m, n, w, seed):
    """[A11 A12; 0 w A22], the heavy rows among the others: weighted constraints that do
    not involve the first columns."""
    A, _ = workloads.gaussian(m, n, seed=seed)
    A = np.array(A)
    rows = np.random.default_rng(seed).choice(np.arange(LIGHT, m), m // 3, replace=False)
    A[rows] *= w
    A[rows, :LIGHT] = 0.0
    return A


def light_rows_error(A, F, up):
    """R12, rows of the light reflectors, against those reflectors applied to A12 in
    extended precision."""
    want = apply_q(F[:, :LIGHT], up[:LIGHT], A[:, LIGHT:], transpose=True)[:LIGHT]
    return float(np.abs(F[:LIGHT, LIGHT:] - want).max() / np.abs(A[:LIGHT]).max())


def factor(c, A, stacked=False):
    m, n = A.shape
    Ad = dev(A)
    up = torch.empty(n, dtype=torch.float64, device="cuda")
    wy = c.wy_buffer(m, n)
    (c.factor_stacked if stacked else c.factor)(Ad, up, wy)
    assert c.sync() == 0
    return Ad, up, wy


SHAPES = [(330, 270), (300, 200), (1100, 192)]


@pytest.mark.parametrize("w", WEIGHTS)
@pytest.mark.parametrize("h", [1, 20, 100])
@pytest.mark.parametrize("m,n", SHAPES)
def test_factor_heavy_rows_on_top(ctx, m, n, h, w):  # noqa: F811
    A = heavy_top(m, n, h, w, h)
    Fo, upo, _ = oracle.h12_factor(A)
    Ad, up, _ = factor(ctx, A)
    report(f"factor {m}x{n} h={h}", w, row_errors(A, Fo, upo).max(),
           row_errors(A, host(Ad), host(up)).max(), n)


@pytest.mark.parametrize("w", WEIGHTS)
@pytest.mark.parametrize("m,n", SHAPES)
def test_factor_heavy_rows_without_the_first_columns(ctx, m, n, w):  # noqa: F811
    A = block_sparse(m, n, w, 5)
    Fo, upo, _ = oracle.h12_factor(A)
    Ad, up, _ = factor(ctx, A)
    report(f"block {m}x{n}", w, light_rows_error(A, Fo, upo),
           light_rows_error(A, host(Ad), host(up)), n)


@pytest.mark.parametrize("w", WEIGHTS)
@pytest.mark.parametrize("n,m_eq", [(300, 150), (280, 20)])
def test_factor_stacked(ctx, n, m_eq, w):  # noqa: F811
    """Rows of L spread over w, in any order."""
    A, _ = workloads.slsqp_stack(n, m_eq, seed=n)
    A = np.array(A)
    A[:n] *= (w ** np.random.default_rng(n).uniform(0.0, 1.0, n))[:, None]
    Fo, upo, _ = oracle.h12_factor(A)
    Ad, up, _ = factor(ctx, A, stacked=True)
    report(f"stacked {n}+{m_eq}", w, row_errors(A, Fo, upo).max(),
           row_errors(A, host(Ad), host(up)).max(), n)


@pytest.mark.parametrize("w", WEIGHTS)
@pytest.mark.parametrize("nrhs", [16, 70])
@pytest.mark.parametrize("use_wy", [True, False])
def test_apply_qt(ctx, nrhs, use_wy, w):  # noqa: F811
    m, n = 330, 270
    A = heavy_top(m, n, 20, w, 6)
    B = heavy_top(m, nrhs, 20, w, 7)
    Ad, up, wy = factor(ctx, A)
    Bd = dev(B)
    ctx.apply_qt(Ad, up, Bd, wy=wy if use_wy else None)
    assert ctx.sync() == 0
    F, u = host(Ad), host(up)
    want = apply_q(F, u, B, transpose=True)
    alpha = np.maximum(np.abs(A).max(axis=1), np.abs(B).max(axis=1))
    alpha = np.maximum(alpha, np.abs(want).max(axis=1))
    one = np.stack([oracle.apply_qt(F, u, np.ascontiguousarray(B[:, j])) for j in range(nrhs)], 1)
    eo, eg = (float((np.abs(v - want).max(axis=1) / alpha).max()) for v in (one, host(Bd)))
    report(f"qt nrhs={nrhs} wy={use_wy}", w, eo, eg, n)


def batch_factor(c, A, copies=1):
    from paper_2506_09463_gb300 import abi
    m, n = A.shape
    Ad = [dev(A) for _ in range(copies)]
    bd = torch.ones(copies, m, dtype=torch.float64, device="cuda")
    up = torch.zeros(copies, n, dtype=torch.float64, device="cuda")
    st = abi.slqr_batch_factor(c.ctx, [m] * copies, [n] * copies, [a.data_ptr() for a in Ad],
                               [m] * copies, [v.data_ptr() for v in up],
                               [v.data_ptr() for v in bd], abi.SLQR_FP64, None, None,
                               torch.cuda.current_stream().cuda_stream)
    abi.check(c.ctx, st, "slqr_batch_factor")
    assert c.sync() == 0
    return host(Ad[0]), host(up[0])


# (400 problems of up to 128 rows and 200 of up to 256 run on the smaller CTAs)
@pytest.mark.parametrize("w", WEIGHTS)
@pytest.mark.parametrize("m,n,h,copies", [(100, 60, 5, 400), (250, 120, 20, 200),
                                          (500, 200, 20, 1), (128, 128, 40, 400)])
def test_batch_heavy_rows_on_top(ctx, m, n, h, copies, w):  # noqa: F811
    A = heavy_top(m, n, h, w, 8)
    Fo, upo, _ = oracle.h12_factor(A)
    F, up = batch_factor(ctx, A, copies)
    report(f"batch {m}x{n} h={h}", w, row_errors(A, Fo, upo).max(), row_errors(A, F, up).max(), n)


@pytest.mark.parametrize("w", WEIGHTS)
@pytest.mark.parametrize("m,n,copies", [(250, 120, 200), (500, 200, 1)])
def test_batch_heavy_rows_without_the_first_columns(ctx, m, n, copies, w):  # noqa: F811
    A = block_sparse(m, n, w, 9)
    Fo, upo, _ = oracle.h12_factor(A)
    F, up = batch_factor(ctx, A, copies)
    report(f"batch block {m}x{n}", w, light_rows_error(A, Fo, upo),
           light_rows_error(A, F, up), n)


@pytest.mark.parametrize("w", WEIGHTS)
@pytest.mark.parametrize("n,m_eq", [(60, 3), (98, 40), (300, 150), (40, 0)])
def test_batch_stacked(ctx, n, m_eq, w):  # noqa: F811
    """Rows of L spread over w, in any order, over few rows of C and many."""
    from paper_2506_09463_gb300 import abi
    A, _ = workloads.slsqp_stack(n, m_eq, seed=n)
    A = np.array(A)
    A[:n] *= (w ** np.random.default_rng(n).uniform(0.0, 1.0, n))[:, None]
    Fo, upo, _ = oracle.h12_factor(A)
    Ad, up = dev(A), torch.zeros(n, dtype=torch.float64, device="cuda")
    st = abi.slqr_batch_factor_stacked(ctx.ctx, [n], [m_eq], [Ad.data_ptr()], [n + m_eq],
                                       [up.data_ptr()], None, abi.SLQR_FP64, None, None,
                                       torch.cuda.current_stream().cuda_stream)
    abi.check(ctx.ctx, st, "slqr_batch_factor_stacked")
    assert ctx.sync() == 0
    report(f"batch stacked {n}+{m_eq}", w, row_errors(A, Fo, upo).max(),
           row_errors(A, host(Ad), host(up)).max(), n)
