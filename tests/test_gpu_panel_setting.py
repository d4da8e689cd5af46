"""slqr_set_panel_cluster for FP64 panels of width 64: only setting 0 takes the panel in
registers.  Which kernel ran shows in the bits: the same sums in another order."""
import pytest
import torch

from test_gpu_fp64_tc import ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(900, 300), (3000, 300)])
def test_setting_takes_effect(ctx, m, n):  # noqa: F811
    from paper_2506_09463_gb300 import abi
    g = torch.Generator(device="cuda").manual_seed(m)
    A0 = torch.randn(n, m, generator=g, dtype=torch.float64, device="cuda").t()
    out = {}
    try:
        for s in (0, -1, 2):
            assert abi.slqr_set_panel_cluster(s) == abi.SLQR_OK
            A = A0.t().clone().t()
            ctx.factor(A)
            assert ctx.sync() == 0
            out[s] = A
    finally:
        assert abi.slqr_set_panel_cluster(0) == abi.SLQR_OK
    assert not torch.equal(out[0], out[-1])
    # two CTAs hold no panel of these rows in shared memory, so setting 2 is the
    # cooperative panel too until the last panels fit
    assert not torch.equal(out[0][:, :64], out[2][:, :64])
    assert torch.equal(out[-1][:, :64], out[2][:, :64])
    # either way the factorization of the same matrix
    assert (out[0] - out[-1]).abs().max() <= 1e-11 * out[0].abs().max()
