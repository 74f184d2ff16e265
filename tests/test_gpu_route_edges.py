"""Operators and gather-scatter on both sides of the sizes at which another kernel
takes over: the same bars on either side (dssum within the rounding of 8 terms of
the oracle and equal for aligned and unaligned vectors)."""
import numpy as np
import pytest

from helpers import pair, torch_dev
from paper_2608_24348_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nel", [(25, 25, 26), (26, 26, 25)])  # 16250 and 16900 unique nodes
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_dssum_of_the_lowest_order(sem, nel, dtype):
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, 1, nel, 0.0)
    u = inputs.local_uniform_field(ctx.nL)
    t = torch.float64 if dtype == "f64" else torch.float32
    a = torch.from_numpy(u).to(dev, t)
    b = torch.empty(ctx.nL + 1, dtype=t, device=dev)[1:]
    b.copy_(a)
    ref = m.dssum(a.cpu().numpy().astype(np.float64))
    ctx.dssum(a, dtype)
    ctx.dssum(b, dtype)
    assert torch.equal(a, b)
    tol = 8 * (1e-15 if dtype == "f64" else 1e-6)
    assert np.abs(a.cpu().numpy().astype(np.float64) - ref).max() <= tol * np.abs(ref).max()
