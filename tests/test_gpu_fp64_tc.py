"""The FP64 trailing update and Q^T B on the tensor cores by exact splitting
(csrc/tc_fp64.cu; panels of 64 reflectors, at least 16 columns) against the
CPU oracle, at the edges of its tiles (128 rows, 32 and 128 columns, 32-row
chunks), and against the FP64-pipe kernels, which a context takes whose budget
does not hold the digit images, also where values are not finite.  Tolerances are those of tests/test_gpu_parity.py.
"""
import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_parity import U, check_against_oracle, dev, factor_tol, host, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2506_09463_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


# (rows, columns, padding of the leading dimension): trailing widths of 16, 17,
# 31..33 and 127..129 columns, row counts around multiples of 32 and 128, odd
# leading dimensions (8-byte loads)
SHAPES = [(337, 336, 0), (384, 273, 0), (385, 287, 1), (513, 289, 0), (449, 449, 3),
          (640, 320, 0), (641, 383, 1), (1023, 385, 0), (1155, 271, 2)]


@pytest.mark.parametrize("m,n,pad", SHAPES)
def test_factor_at_tile_edges(ctx, m, n, pad):
    A, b = workloads.gaussian(m, n, seed=m + n)
    F, up, qtb, x, st = run_gpu(ctx, A, b, lda_pad=pad)
    assert st == 0
    check_against_oracle(A, b, F, up, qtb, x)


@pytest.mark.parametrize("nrhs", [15, 16, 17, 33, 64, 130])
@pytest.mark.parametrize("stacked", [False, True])
def test_apply_qt_blocks(ctx, nrhs, stacked):
    if stacked:
        n, m = 300, 450
        A, _ = workloads.slsqp_stack(n, m - n, seed=nrhs)
    else:
        m, n = 461, 300
        A, _ = workloads.gaussian(m, n, seed=nrhs)
    B = workloads.gaussian_rhs(m, nrhs, seed=nrhs)
    Ad, Bd = dev(A), dev(B)
    up = torch.empty(n, dtype=torch.float64, device="cuda")
    wy = ctx.wy_buffer(m, n)
    (ctx.factor_stacked if stacked else ctx.factor)(Ad, up, wy)
    (ctx.apply_qt_stacked if stacked else ctx.apply_qt)(Ad, up, Bd, wy=wy)
    assert ctx.sync() == 0
    Fo, upo, _ = oracle.h12_factor(A)
    _, kappa = factor_tol(A)
    out = host(Bd)
    for j in range(nrhs):
        want = oracle.apply_qt(Fo, upo, np.ascontiguousarray(B[:, j]))
        np.testing.assert_allclose(out[:, j], want, rtol=0,
                                   atol=4.0 * np.sqrt(m) * U * kappa * np.linalg.norm(B[:, j]))


def test_columns_of_any_scale(ctx):
    """Powers of two per column are exact: the factorization of A D is F D."""
    m, n = 500, 360
    A, b = workloads.gaussian(m, n, seed=5)
    e = np.random.default_rng(6).integers(-450, 451, size=n)
    F, up, _, _, st = run_gpu(ctx, A, b)
    assert st == 0
    G, upg, _, _, st = run_gpu(ctx, np.ldexp(A, e[None, :]), b)
    assert st == 0
    tol, _ = factor_tol(A)
    np.testing.assert_allclose(np.ldexp(G, -e[None, :]), F, rtol=0, atol=tol)
    np.testing.assert_allclose(np.ldexp(upg, -e), up, rtol=0, atol=tol)


# a budget that holds the workspace of the FP64-pipe kernels (68 MB) but not the
# digit images of 20,000 rows (120 MB in all)
PIPE_BUDGET = 90 << 20


@pytest.mark.parametrize("value", [None, np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("row,col", [(3, 130), (19000, 70), (19000, 10)])
def test_same_as_the_fp64_pipe(ctx, value, row, col):
    """Over the budget every update stays on the FP64 pipe: the same values to
    the parity tolerance, and not finite in the same places."""
    from paper_2506_09463_gb300 import api
    m, n = 20000, 300
    A, b = workloads.gaussian(m, n, seed=8)
    A = np.array(A)
    if value is not None:
        A[row, col] = value
    F, up, _, _, _ = run_gpu(ctx, A, b)
    with api.Context(0, hbm_budget_bytes=PIPE_BUDGET) as pipe:
        G, upg, _, _, _ = run_gpu(pipe, A, b)
    np.testing.assert_array_equal(np.isfinite(up), np.isfinite(upg))
    np.testing.assert_array_equal(np.isfinite(F), np.isfinite(G))
    if value is None:
        tol, _ = factor_tol(A)
        np.testing.assert_allclose(F, G, rtol=0, atol=tol)
        assert not np.array_equal(F, G)          # (the two paths round differently)


# right-hand sides of one launch (1, 2, 4) and remainders; rows per CTA 32, 64,
# 128 with one cluster and several; panels of 32 and 64, a ragged last one
@pytest.mark.parametrize("m,n", [(200, 150), (700, 321), (2200, 130), (4300, 260), (8300, 70)])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 5, 15])
@pytest.mark.parametrize("use_wy", [True, False])
def test_apply_qt_few_right_hand_sides(ctx, m, n, nrhs, use_wy):
    A, _ = workloads.gaussian(m, n, seed=m + nrhs)
    B = workloads.gaussian_rhs(m, nrhs, seed=nrhs)
    Ad, Bd = dev(A), dev(B)
    up = torch.empty(n, dtype=torch.float64, device="cuda")
    wy = ctx.wy_buffer(m, n) if use_wy else None
    ctx.factor(Ad, up, wy)
    ctx.apply_qt(Ad, up, Bd, wy=wy)
    ctx.solve_r(Ad, Bd)
    assert ctx.sync() == 0
    F, upf, out = host(Ad), host(up), host(Bd)
    for j in range(nrhs):
        b = np.ascontiguousarray(B[:, j])
        qtb = oracle.apply_qt(F, upf, b)
        x, _ = oracle.solve_r(F, qtb)
        # the same factorization applied: Q^T b to the summation's rounding, x by
        # the condition of R
        np.testing.assert_allclose(out[n:, j], qtb[n:], rtol=0,
                                   atol=4.0 * np.sqrt(m) * U * np.linalg.norm(b) * np.sqrt(n))
        kappa = np.linalg.cond(np.triu(F[:n]))
        assert np.linalg.norm(out[:n, j] - x) <= 64.0 * kappa * U * np.sqrt(n) * \
            np.linalg.norm(b) / np.linalg.norm(A, 2) + 64.0 * kappa * U * np.linalg.norm(x)


@pytest.mark.parametrize("m,n", [(64, 32), (70, 69), (256, 128), (300, 200), (257, 256)])
def test_compact_wy_of_few_columns(ctx, m, n):
    """Panels of 32 in the store, factored in panels of 64: the store's blocks against
    V of the factorization (G = striu(V^T V), tau = -1 / (up R_kk))."""
    A, _ = workloads.gaussian(m, n, seed=m)
    Ad = dev(A)
    up = torch.empty(n, dtype=torch.float64, device="cuda")
    wy = ctx.wy_buffer(m, n)
    wy.fill_(float("nan"))
    ctx.factor(Ad, up, wy)
    assert ctx.sync() == 0
    F, u, store = host(Ad), host(up), host(wy)
    K = min(m - 1, n)
    V = np.tril(F, -1)[:, :K] + np.vstack([np.diag(u[:K]), np.zeros((m - K, K))])
    size = 2 * 32 * 32 + 32
    for p in range((K + 31) // 32):
        k0, w = 32 * p, min(32, K - 32 * p)
        blk = store[p * size:(p + 1) * size]
        Vp = V[k0:, k0:k0 + w]
        vtop = blk[:1024].reshape(32, 32).T
        np.testing.assert_array_equal(vtop[:min(w, m - k0), :w], Vp[:w][:, :w])
        G = blk[1024:2048].reshape(32, 32).T[:w, :w]
        want = np.triu(Vp.T @ Vp, 1)
        nrm = np.linalg.norm(Vp, axis=0)
        assert np.all(np.abs(np.triu(G, 1) - want) <= 4.0 * np.sqrt(m) * U * np.outer(nrm, nrm))
        tau = -1.0 / (u[k0:k0 + w] * np.diag(F)[k0:k0 + w])
        np.testing.assert_allclose(blk[2048:2048 + w], tau, rtol=16 * U)


# the last rows of one cluster of 16 CTAs of 32 and of 80 rows, clusters of 8 with
# up to 10 and with more sums to collect, clusters of 4; a last panel of 1..6 columns
@pytest.mark.parametrize("m,n", [(33, 33), (512, 70), (513, 65), (1280, 130), (1281, 67),
                                 (2049, 66), (16385, 69), (21000, 70), (29000, 68)])
def test_panel_shapes(ctx, m, n):
    A, b = workloads.gaussian(m, n, seed=m - n)
    F, up, qtb, x, st = run_gpu(ctx, A, b)
    assert st == 0
    check_against_oracle(A, b, F, up, qtb, x)


# back-substitution of few right-hand sides in one launch: one row block, a ragged
# last one, several, and more than are resident at once; zero and not finite
# diagonal entries
@pytest.mark.parametrize("n", [64, 65, 127, 129, 640, 2049, 9800])
@pytest.mark.parametrize("nrhs", [1, 3, 4, 5])
@pytest.mark.parametrize("kind", ["plain", "zero", "nan"])
def test_solve_r_few_right_hand_sides(ctx, n, nrhs, kind):
    g = torch.Generator(device="cuda").manual_seed(n + nrhs)
    R = torch.randn(n, n, generator=g, dtype=torch.float64, device="cuda") / n ** 0.5   # R^T
    R.diagonal().copy_(2.0 + torch.rand(n, generator=g, dtype=torch.float64, device="cuda"))
    B0 = torch.randn(nrhs, n, generator=g, dtype=torch.float64, device="cuda")
    k = n // 2
    if kind == "zero":
        R[k, k] = 0.0
    if kind == "nan":
        R[n - 1, n - 1] = float("nan")
    B = B0.clone()
    ctx.solve_r(R.T, B.T)
    st = ctx.sync()
    U_ = torch.triu(R.T)
    if kind == "nan":
        assert torch.isnan(B).all()
        return
    assert st == (0 if kind == "plain" else ctx_rank())
    if kind == "zero":                             # x_k = 0, the other equations hold
        assert (B[:, k] == 0).all()
        U_[k, k] = 1.0
        B0[:, k] = (U_[k, k + 1:] @ B[:, k + 1:].T)
    # row-wise backward error of the blocks' products: 64 + n terms, the block inverses
    # with condition below (1 + 64 max |R_ij| / 2)^2 of well-scaled rows
    res = (U_ @ B.T - B0.T).abs()
    scale = U_.abs() @ B.T.abs() + B0.T.abs()
    assert (res <= (n + 64) * 16 * U * scale).all()


def ctx_rank():
    from paper_2506_09463_gb300 import abi
    return abi.SLQR_ERANK
