"""Where a value that is not finite may go in the FP64 kernels for few right-hand sides.

Back-substitution: row c of the right-hand sides reaches rows up to c only, so the rows
below are, bit for bit, those of the same call with a finite value there.  Q^T b of a
stacked [L^T; C]: a row of the top block meets the reflectors of its own panel and later
ones only.
"""
import numpy as np
import pytest
import torch

import workloads
from test_gpu_fp64_tc import ctx  # noqa: F401
from test_gpu_parity import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("n,row", [(50, 7), (64, 0), (130, 70), (130, 128), (640, 200)])
@pytest.mark.parametrize("nrhs", [1, 3, 5, 64])
def test_solve_r_leaves_the_rows_below(ctx, n, row, nrhs, value):  # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(n + nrhs)
    R = torch.randn(n, n, generator=g, dtype=torch.float64, device="cuda") / n ** 0.5   # R^T
    R.diagonal().copy_(2.0 + torch.rand(n, generator=g, dtype=torch.float64, device="cuda"))
    B = torch.randn(nrhs, n, generator=g, dtype=torch.float64, device="cuda")
    clean, bad = B.clone(), B.clone()
    bad[nrhs - 1, row] = value
    ctx.solve_r(R.T, clean.T)
    ctx.solve_r(R.T, bad.T)
    assert ctx.sync() == 0
    assert torch.equal(bad[:, row + 1:], clean[:, row + 1:])
    assert torch.equal(bad[:nrhs - 1], clean[:nrhs - 1])
    assert not torch.isfinite(bad[nrhs - 1, row])


# the row shares a CTA (32 or 64 rows) with rows of C, or with another panel of 32
@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("n,m_eq,row,nb", [(300, 150, 290, 64), (200, 2000, 40, 32),
                                           (250, 4100, 100, 32)])
@pytest.mark.parametrize("nrhs", [1, 2, 4])
def test_apply_qt_stacked_leaves_earlier_panels(ctx, n, m_eq, row, nb, nrhs, value):  # noqa: F811
    A, _ = workloads.slsqp_stack(n, m_eq, seed=n)
    B = workloads.gaussian_rhs(n + m_eq, nrhs, seed=nrhs)
    Ad, clean, bad = dev(A), dev(B), dev(B)
    bad[row, nrhs - 1] = value
    up = torch.empty(n, dtype=torch.float64, device="cuda")
    wy = ctx.wy_buffer(n + m_eq, n)
    ctx.factor_stacked(Ad, up, wy)
    ctx.apply_qt_stacked(Ad, up, clean, wy=wy)
    ctx.apply_qt_stacked(Ad, up, bad, wy=wy)
    assert ctx.sync() == 0
    first = row // nb * nb                       # rows of the panels before
    assert torch.equal(bad[:first], clean[:first])
    assert torch.equal(bad[:, :nrhs - 1], clean[:, :nrhs - 1])
    assert not torch.isfinite(bad[row:, nrhs - 1]).any()
