"""Split-operand tensor-core operator at even orders (odd N+1), whose slabs do not
fill a multiple of 16 bytes: eight elements and more a block, the FP32 operator's
bar of 1e-5 of the largest output of an element, and the solve around it."""
import numpy as np
import pytest

from helpers import fourier_rhs, pair, torch_dev
from paper_2608_24348_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f16x2_tc", "bf16x3_tc"])
@pytest.mark.parametrize("N", [2, 4, 6])
def test_split_operands_at_even_orders(sem, dtype, N):
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, N, (3, 2, 3), 0.1)
    u = inputs.local_uniform_field(ctx.nL, seed=7).astype(np.float32)
    ref = m.ax(u.astype(np.float64), 0.01, 1000.0).reshape(ctx.E, -1)
    ud = torch.from_numpy(u).to(dev)
    wd = torch.empty_like(ud)
    ctx.ax(ud, wd, 0.01, 1000.0, dtype)
    got = wd.cpu().numpy().astype(np.float64).reshape(ctx.E, -1)
    for e in range(ctx.E):
        assert np.abs(got[e] - ref[e]).max() <= 1e-5 * np.abs(ref[e]).max(), (N, e)


@pytest.mark.parametrize("dtype", ["f16x2_tc", "bf16x3_tc"])
@pytest.mark.parametrize("N", [2, 4, 6])
def test_solve_with_split_operands_at_even_orders(sem, dtype, N):
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, N, (4, 3, 3), 0.1)
    bg, bo = fourier_rhs(ctx, m)
    x = torch.zeros_like(bg)
    info = ctx.pcg_solve(bg, x, 1.0, 2.0, tol=1e-10, inner=dtype)
    assert info["status"] == 0, info
    r, bn = m.residual(bo, x.cpu().numpy(), 1.0, 2.0)
    assert r <= 1.5e-10 * bn, (r, bn)
