"""The polled exchanges of Q^T b (csrc/qt_vec.cu) and of the back-substitution of few
right-hand sides (csrc/solve.cu) under a short spin limit: SLQR_ETIMEOUT is reported, and
the same context gives the same results as before at the default limit."""
import pytest
import torch

from test_gpu_fp64_tc import ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["apply_qt", "solve_r"])
def test_short_limit_is_reported(ctx, call):  # noqa: F811
    from paper_2506_09463_gb300 import abi
    m, n = 3000, 1000                            # 24 CTAs in clusters; 16 row blocks
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn(n, m, generator=g, dtype=torch.float64, device="cuda").t()
    b = torch.randn(1, m, generator=g, dtype=torch.float64, device="cuda").t()
    up = torch.empty(n, dtype=torch.float64, device="cuda")
    wy = ctx.wy_buffer(m, n)
    ctx.factor(A, up, wy)

    def run():
        x = b.clone()
        if call == "apply_qt":
            ctx.apply_qt(A, up, x, wy=wy)
        else:
            ctx.solve_r(A, x)
        return x, ctx.sync()

    want, st = run()
    assert st == 0
    try:
        assert abi.slqr_set_spin_limit(ctx.ctx, 1) == abi.SLQR_OK
        seen = [run()[1] for _ in range(3)]      # (the CTAs' arrival order is not fixed)
        assert abi.SLQR_ETIMEOUT in seen, seen
        assert all(s in (abi.SLQR_OK, abi.SLQR_ETIMEOUT) for s in seen), seen
    finally:
        assert abi.slqr_set_spin_limit(ctx.ctx, 0) == abi.SLQR_OK
    x, st = run()
    assert st == 0 and torch.equal(x, want)
