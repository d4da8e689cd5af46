"""The mixed-precision batch (SLQR_FP32: FP32 factorization, FP64 refinement) at
the edges of its column scaling, its status of values that are not finite, and
within a budget that holds the scratch of two CTAs to an SM, not of three.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

BUDGET = 450 << 20          # (456 CTAs take 544 MB, 304 take 363)


def _problems(count, seed, m_hi=60):
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(count):
        m = int(rng.integers(2, m_hi + 1))
        n = int(rng.integers(1, m + 1))
        A = rng.standard_normal((m, n))
        A[np.arange(n), np.arange(n)] += 2.0 * np.sqrt(m)
        out.append((A, rng.standard_normal(m)))
    return out


def _solve(problems, plan=False, budget=0):
    from paper_2506_09463_gb300 import abi, api
    dev = [torch.from_numpy(np.ascontiguousarray(A.T)).cuda() for A, _ in problems]
    bs = [torch.from_numpy(b.copy()).cuda() for _, b in problems]
    status = torch.full((len(problems),), 99, dtype=torch.int32, device="cuda")
    err = torch.zeros(len(problems), dtype=torch.float64, device="cuda")
    ms, ns = [A.shape[0] for A, _ in problems], [A.shape[1] for A, _ in problems]
    with api.Context(0, hbm_budget_bytes=budget) as ctx:
        args = (ms, ns, [d.data_ptr() for d in dev], ms, None, [b.data_ptr() for b in bs],
                abi.SLQR_FP32, status.data_ptr(), err.data_ptr())
        if plan:
            st, h = abi.slqr_batch_plan_create(ctx.ctx, ms, ns, None, *args[2:])
            abi.check(ctx.ctx, st, "slqr_batch_plan_create")
            abi.check(ctx.ctx, abi.slqr_batch_plan_launch(h, 0), "slqr_batch_plan_launch")
            torch.cuda.synchronize()
            abi.slqr_batch_plan_destroy(h)
        else:
            abi.check(ctx.ctx, abi.slqr_batch_factor(ctx.ctx, *args, 0), "slqr_batch_factor")
            ctx.sync()
    return [b.cpu().numpy() for b in bs], status.cpu().numpy(), err.cpu().numpy()


@pytest.mark.parametrize("plan", [False, True])
def test_within_a_budget_of_two_ctas_to_an_sm(plan):
    problems = _problems(500, seed=1)
    x, st, _ = _solve(problems, plan)
    y, st2, _ = _solve(problems, plan, BUDGET)
    assert np.all(st == 0) and np.all(st2 == 0)
    for a, b in zip(x, y):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("e", [0, 900, -900, -1015])
def test_columns_of_any_scale(e):
    """Powers of two are exact up to the rounding of subnormal entries, 2^-59 of the
    largest at 2^-1015.  The refinement stops at steps of 1e-14 of x, contracting by
    more than a half: 4e-14 of the solution, and the solution error of the problem,
    64 (kappa + kappa^2 ||r|| / (||A|| ||x||)) 2^-53."""
    for A, b in _problems(20, seed=2):
        (x,), st, _ = _solve([(np.ldexp(A, e), b)])
        assert st[0] == 0
        n = A.shape[1]
        xo, _, _, qtb, _ = oracle.lstsq(A, b)
        kappa, r = np.linalg.cond(A), oracle.residual_norm(qtb, n)
        bound = 4e-14 + 64 * (kappa + kappa ** 2 * r / (np.linalg.norm(A, 2) * np.linalg.norm(xo))) * 2.0 ** -53
        assert np.linalg.norm(np.ldexp(x[:n], e) - xo) <= bound * np.linalg.norm(xo)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_not_finite_is_reported(value):
    from paper_2506_09463_gb300 import abi
    problems = _problems(6, seed=3)
    for A, _ in problems[::2]:
        A[A.shape[0] // 2, A.shape[1] // 2] = value
    _, st, err = _solve(problems)
    assert np.all(st[::2] == abi.SLQR_ENOCONV) and np.all(np.isinf(err[::2]))
    assert np.all(st[1::2] == 0)
