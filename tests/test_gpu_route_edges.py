"""Operators and gather-scatter on both sides of the sizes at which another kernel
takes over: the same bars on either side (dssum within the rounding of 8 terms of
the oracle and equal for aligned and unaligned vectors; FP32 operator 1e-5 of the
largest output, for the built-in choice and for candidate 0, on meshes of one and of
several waves of blocks)."""
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


@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 7, 8, 9, 10, 13])
@pytest.mark.parametrize("shift", [1, 2, 4])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_dssum_of_shifted_vectors(sem, N, shift, dtype):
    """Vectors that start one, two and four values past an aligned address: chunks
    take as many values at a time as the order allows, so each shift is aligned for
    some orders and not for others."""
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, N, (3, 3, 2), 0.0)
    u = inputs.local_uniform_field(ctx.nL)
    t = torch.float64 if dtype == "f64" else torch.float32
    a = torch.from_numpy(u).to(dev, t)
    base = torch.full((ctx.nL + shift + 8,), 7.0, dtype=t, device=dev)
    b = base[shift:shift + ctx.nL]
    b.copy_(a)
    ref = m.dssum(a.cpu().numpy().astype(np.float64))
    ctx.dssum(a, dtype)
    ctx.dssum(b, dtype)
    assert torch.equal(a, b)
    assert bool((base[:shift] == 7.0).all()) and bool((base[shift + ctx.nL:] == 7.0).all())
    tol = 8 * (1e-15 if dtype == "f64" else 1e-6)
    assert np.abs(a.cpu().numpy().astype(np.float64) - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("N,nel", [(2, (1, 1, 1)), (2, (13, 12, 13)), (6, (8, 9, 10)), (6, (9, 9, 10)), (7, (8, 8, 9)),
                                   (7, (9, 9, 8)), (8, (8, 8, 8)), (9, (8, 8, 9)), (9, (9, 9, 8)), (10, (8, 8, 8)),
                                   (11, (8, 8, 8)), (12, (8, 8, 8)), (13, (9, 10, 10)), (13, (9, 10, 11)),
                                   (14, (6, 7, 6)), (15, (6, 7, 6))])
def test_fp32_operator(sem, N, nel):
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, N, nel, 0.1)
    u = torch.from_numpy(inputs.local_uniform_field(ctx.nL)).to(dev).float()
    ref = m.ax(u.cpu().numpy().astype(np.float64), 0.3, 2.0)
    w = torch.empty_like(u)
    for variant in (-1, 0):
        w.fill_(float("nan"))
        sem.set_ax_variant(N, "f32", variant)
        try:
            ctx.ax(u, w, 0.3, 2.0, "f32")
        finally:
            sem.set_ax_variant(N, "f32", -1)
        assert np.abs(w.cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max(), variant
