"""Q^T B of fewer than 16 right-hand sides on both sides of the rule that chooses between
one launch for all panels and the tiled products (one and two panels, up to two and more
launches), against the oracle's application of the same reflectors."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_fp64_tc import ctx  # noqa: F401
from test_gpu_parity import U, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(40, 20), (64, 32), (100, 64), (9000, 30)])
@pytest.mark.parametrize("nrhs", [4, 8, 9, 15])
def test_few_panels(ctx, m, n, nrhs):  # noqa: F811
    A, _ = workloads.gaussian(m, n, seed=m)
    B = workloads.gaussian_rhs(m, nrhs, seed=nrhs)
    Ad, Bd = dev(A), dev(B)
    up = torch.empty(n, dtype=torch.float64, device="cuda")
    wy = ctx.wy_buffer(m, n)
    ctx.factor(Ad, up, wy)
    ctx.apply_qt(Ad, up, Bd, wy=wy)
    assert ctx.sync() == 0
    F, upf, out = host(Ad), host(up), host(Bd)
    for j in range(nrhs):
        b = np.ascontiguousarray(B[:, j])
        np.testing.assert_allclose(out[:, j], oracle.apply_qt(F, upf, b), rtol=0,
                                   atol=4.0 * np.sqrt(m * n) * U * np.linalg.norm(b))
