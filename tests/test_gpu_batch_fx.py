"""The batched FP64 factorization on the tensor cores (csrc/batch_fx.cu, the
default setting) at the edges of its three kernels (problems of up to 128, 256
and 512 rows; panels of 16 reflectors, column tiles of 8) against the CPU oracle,
and against the FP64-pipe kernel of another setting where columns are of extreme
scale or values are not finite.  Tolerances are those of tests/test_gpu_batch.py.
"""
import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_batch import U, check_problem, ctx, problem, run_batch  # noqa: F401

pytestmark = pytest.mark.gpu

# problems of one launch: the largest row count and the number of problems (at most
# 152, 304, more) pick the kernel
COPIES = [1, 20, 40]
LAUNCHES = {
    128: [(128, 128), (128, 127), (127, 16), (127, 17), (128, 15), (126, 9), (33, 32), (16, 15)],
    256: [(129, 129), (255, 31), (256, 256), (256, 33), (129, 8), (130, 7), (7, 7), (1, 1)],
    512: [(257, 257), (511, 16), (511, 17), (512, 511), (512, 15), (300, 64), (24, 24), (15, 0)],
}


@pytest.mark.parametrize("copies", COPIES)
@pytest.mark.parametrize("rows", sorted(LAUNCHES))
def test_edges_against_oracle(ctx, rows, copies):  # noqa: F811
    ms, ns = zip(*LAUNCHES[rows] * copies)
    res = run_batch(ctx, ms, ns, seed=rows)
    assert np.all(res["status"] == 0)
    for i, (m, n) in enumerate(LAUNCHES[rows]):
        check_problem(*problem(res, i, m, n))


@pytest.mark.parametrize("copies", COPIES)
@pytest.mark.parametrize("rows", sorted(LAUNCHES))
def test_factor_only(ctx, rows, copies):  # noqa: F811
    ms, ns = zip(*LAUNCHES[rows] * copies)
    res = run_batch(ctx, ms, ns, seed=rows + 1, with_b=False)
    for i, (m, n) in enumerate(LAUNCHES[rows]):
        if n == 0:
            continue
        A0, F, b0, b, up = problem(res, i, m, n)
        F_o, up_o, _ = oracle.h12_factor(A0)
        tol = 4.0 * np.sqrt(m) * U * np.linalg.cond(A0) * float(np.linalg.norm(A0, axis=0).max())
        np.testing.assert_allclose(F, F_o, rtol=0, atol=tol)
        np.testing.assert_array_equal(b, b0)


def _factor(ctx, A_list, setting):  # noqa: F811
    from paper_2506_09463_gb300 import abi
    given = len(A_list)
    A_list = A_list + [A_list[0]] * (310 if A_list[0].shape[0] < 256 else 0)   # (every kernel)
    count = len(A_list)
    dev = [torch.from_numpy(np.asfortranarray(A).T.copy()).cuda() for A in A_list]
    ups = [torch.zeros(A.shape[1], dtype=torch.float64, device="cuda") for A in A_list]
    status = torch.zeros(count, dtype=torch.int32, device="cuda")
    assert abi.slqr_batch_set_tuning(abi.SLQR_FP64, -1, *setting) == abi.SLQR_OK
    try:
        st = abi.slqr_batch_factor(ctx.ctx, [A.shape[0] for A in A_list],
                                   [A.shape[1] for A in A_list], [d.data_ptr() for d in dev],
                                   [A.shape[0] for A in A_list], [u.data_ptr() for u in ups], None,
                                   abi.SLQR_FP64, status.data_ptr(), None,
                                   torch.cuda.current_stream().cuda_stream)
        abi.check(ctx.ctx, st, "slqr_batch_factor")
        ctx.sync()
    finally:
        assert abi.slqr_batch_set_tuning(abi.SLQR_FP64, -1, 0, 0) == abi.SLQR_OK
    return [d.cpu().numpy().T for d in dev[:given]], [u.cpu().numpy() for u in ups[:given]]


@pytest.mark.parametrize("span", [450, 960])
@pytest.mark.parametrize("rows", sorted(LAUNCHES))
def test_columns_of_any_scale(ctx, rows, span):  # noqa: F811
    """Powers of two per column are exact: the factorization of A D is F D, as long as
    up times the diagonal entry, 2^(2 e), stays in range.  Beyond that the values are
    finite in the same places as with the setting (16, 16)."""
    m, n = rows - 3, min(rows - 5, 90)
    A, _ = workloads.gaussian(m, n, seed=rows + 2)
    e = np.random.default_rng(rows).integers(-span, span, n)
    if span > 500:
        e[:3] = -1000, 900, 0
    D = np.ldexp(A, e[None, :])
    (F, Fd), _ = _factor(ctx, [A, D], (0, 0))
    if span > 500:
        (G,), _ = _factor(ctx, [D], (16, 16))
        np.testing.assert_array_equal(np.isfinite(Fd), np.isfinite(G))
        return
    kappa = np.linalg.cond(A)
    tol = 8.0 * np.sqrt(m) * U * kappa * np.linalg.norm(A, axis=0).max()
    np.testing.assert_allclose(np.ldexp(Fd, -e[None, :]), F, rtol=0, atol=tol)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("rows", sorted(LAUNCHES))
def test_not_finite_as_on_the_fp64_pipe(ctx, rows, value):  # noqa: F811
    """Not finite in the same places as with the setting (16, 16); the columns
    before the value are as without it."""
    m, n = rows - 1, 50
    A, _ = workloads.gaussian(m, n, seed=rows + 3)
    A[rows // 2, 21] = value
    (F,), (up,) = _factor(ctx, [A], (0, 0))
    (G,), (up_g,) = _factor(ctx, [A], (16, 16))
    np.testing.assert_array_equal(np.isfinite(F), np.isfinite(G))
    np.testing.assert_array_equal(np.isfinite(up), np.isfinite(up_g))
    tol = 8.0 * np.sqrt(m) * U * np.linalg.cond(A[:, :21]) * np.linalg.norm(A[:, :21], axis=0).max()
    np.testing.assert_allclose(F[:, :21], G[:, :21], rtol=0, atol=tol)
