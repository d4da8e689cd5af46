"""The scale of a column's norm in the batched FP64 panel (csrc/batch_fx.cu)."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_batch import ctx  # noqa: F401
from test_gpu_parity import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [100, 200, 500])
def test_batch_entries_above_the_diagonal_do_not_scale_the_norm(ctx, rows):  # noqa: F811
    """Upper triangular with entries of 2^700 above the diagonal: every reflector flips
    the sign of its row (R_kk = -A_kk, up = 2 A_kk), as in the oracle."""
    from paper_2506_09463_gb300 import abi
    n = 40
    rng = np.random.default_rng(rows)
    A = np.zeros((rows, n))
    A[:n] = np.triu(rng.uniform(0.5, 2.0, (n, n)))
    A[0, 5] = A[2, 9] = 2.0 ** 700
    Fo, upo, _ = oracle.h12_factor(A)
    assert np.all(upo != 0)
    d = dev(A)
    up = torch.zeros(n, dtype=torch.float64, device="cuda")
    st = abi.slqr_batch_factor(ctx.ctx, [rows], [n], [d.data_ptr()], [rows], [up.data_ptr()], None,
                               abi.SLQR_FP64, None, None, torch.cuda.current_stream().cuda_stream)
    abi.check(ctx.ctx, st, "slqr_batch_factor")
    assert ctx.sync() == 0
    np.testing.assert_allclose(np.diag(host(d)), np.diag(Fo), rtol=2.0 ** -50)
    np.testing.assert_allclose(host(up), upo, rtol=2.0 ** -50)
