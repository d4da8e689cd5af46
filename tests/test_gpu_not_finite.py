"""Where a value that is not finite may go in the FP64 kernels for few right-hand sides.

Back-substitution: row c of the right-hand sides reaches rows up to c only, so the rows
below are, bit for bit, those of the same call with a finite value there.
"""
import numpy as np
import pytest
import torch

from test_gpu_fp64_tc import ctx  # noqa: F401

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
