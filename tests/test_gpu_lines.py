"""GPU checks of the kernels that work by whole lines and of the chunked passes
over the unique nodes, at the sizes where they can go wrong: every order (odd
and even N+1, the largest of each form), single elements and ragged groups,
meshes one element wide, periodic and not, vectors aligned for vector accesses
and not.

Bars: FP64-accurate operator 1e-12 and FP32 operator 1e-5 of the largest output
(those of test_gpu_ops), dssum bit-identical between the two forms and within
the rounding of 8 terms of the oracle, solves to the oracle's residual and 1e-9
of its solution.
"""
import numpy as np
import pytest

from helpers import fourier_rhs, gpu_coords, pair, rel, sine_rhs, torch_dev
from paper_2608_24348_gb300 import inputs

pytestmark = pytest.mark.gpu


def _err(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("N", range(1, 16))
@pytest.mark.parametrize("nel", [(1, 1, 1), (3, 2, 5)])
def test_line_operators_every_order(sem, N, nel):
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, N, nel, 0.1)
    u = inputs.local_uniform_field(ctx.nL)
    ref = m.ax(u, 0.3, 2.0)
    ud = torch.from_numpy(u).to(dev)
    w = torch.empty_like(ud)
    ctx.ax(ud, w, 0.3, 2.0, "f64")
    assert _err(w.cpu().numpy(), ref) <= 1e-12
    u32 = ud.float()
    w32 = torch.empty_like(u32)
    sem.set_ax_variant(N, "f32", 0)
    try:
        ctx.ax(u32, w32, 0.3, 2.0, "f32")
    finally:
        sem.set_ax_variant(N, "f32", -1)
    assert _err(w32.cpu().numpy(), m.ax(u32.cpu().numpy().astype(np.float64), 0.3, 2.0)) <= 1e-5


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 9, 11, 14])
@pytest.mark.parametrize("nel,periodic", [((1, 1, 1), (1, 1, 1)), ((3, 1, 4), (1, 1, 0)), ((1, 3, 2), (0, 1, 1)),
                                          ((4, 3, 2), (0, 0, 0))])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_dssum_forms_agree(sem, N, nel, periodic, dtype):
    """Aligned vectors go by chunks, others one node at a time: the same sums."""
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, N, nel, 0.0, periodic)
    u = inputs.local_uniform_field(ctx.nL)
    t = torch.float64 if dtype == "f64" else torch.float32
    a = torch.from_numpy(u).to(dev, t)
    base = torch.empty(ctx.nL + 1, dtype=t, device=dev)
    b = base[1:]
    b.copy_(a)
    u0 = a.cpu().numpy().astype(np.float64)
    ctx.dssum(a, dtype)
    ctx.dssum(b, dtype)
    assert torch.equal(a, b)
    tol = 1e-15 if dtype == "f64" else 1e-6
    assert _err(a.cpu().numpy().astype(np.float64), m.dssum(u0)) <= 8 * tol


@pytest.mark.parametrize("N,nel,periodic", [(2, (5, 4, 3), (1, 1, 1)), (4, (3, 3, 3), (0, 1, 1)),
                                            (6, (1, 3, 2), (1, 1, 1)), (8, (2, 2, 3), (0, 0, 0)),
                                            (10, (2, 2, 2), (1, 1, 1)), (11, (2, 1, 2), (1, 1, 1)),
                                            (13, (1, 2, 2), (1, 1, 1))])
@pytest.mark.parametrize("inner", ["f64", "f32", "f64_native"])
def test_solve_on_unaligned_vectors(sem, N, nel, periodic, inner):
    """Helmholtz solves whose vectors start 8 bytes past an aligned address take
    the scalar accesses of the caller's vectors: the same bits as aligned ones,
    and the oracle's solution."""
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, N, nel, 0.1, periodic)
    rng = np.random.default_rng(7)
    bo = m.dssum(rng.uniform(-1, 1, ctx.nL))
    xo, info_o = m.pcg(bo, 1.0, 3.0, tol=1e-12)
    out = []
    for shift in (0, 1):
        b = torch.empty(ctx.nL + 1, dtype=torch.float64, device=dev)[shift:shift + ctx.nL]
        x = torch.zeros(ctx.nL + 1, dtype=torch.float64, device=dev)[shift:shift + ctx.nL]
        b.copy_(torch.from_numpy(bo))
        info = ctx.pcg_solve(b, x, 1.0, 3.0, tol=1e-11, inner=inner)
        assert info["status"] == 0, info
        out.append(x.clone())
    assert torch.equal(out[0], out[1])
    assert rel(out[0].cpu().numpy(), xo) <= 1e-9


def test_solve_keeps_a_guess_that_jumps_between_elements(sem):
    """The correction is the same at every copy of a node: an initial guess with
    different values at the copies keeps their differences."""
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, 5, (3, 2, 4), 0.1)
    bg, _, _ = sine_rhs(ctx, m)
    x0 = torch.from_numpy(inputs.local_uniform_field(ctx.nL)).to(dev)
    x = x0.clone()
    assert ctx.pcg_solve(bg, x, 1.0, 2.0, tol=1e-10)["status"] == 0
    d = (x - x0).cpu().numpy()
    mult = m.dssum(np.ones(ctx.nL))
    assert np.abs(m.dssum(d) / mult - d).max() <= 1e-14 * np.abs(x0.cpu().numpy()).max() * 8


@pytest.mark.parametrize("inner", ["f64", "f32"])
def test_batch_shares_the_jacobi_inverse(sem, inner):
    """Problems on one context with the same coefficients use one Jacobi inverse;
    different coefficients keep their own; each solution is that of its own solve,
    and so is a second call's, which finds the inverses cached."""
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, 7, (3, 2, 3), 0.1)
    other, _, _ = pair(sem, 5, (4, 3, 3), 0.1)
    rhs = [torch.from_numpy(m.dssum(np.random.default_rng(s).uniform(-1, 1, ctx.nL))).to(dev) for s in range(3)]
    bo, _, _ = sine_rhs(other, None)
    ctxs, bs, h2 = [ctx, other, ctx, ctx], [rhs[0], bo, rhs[1], rhs[2]], [4.0, 1.0, 4.0, 9.0]
    for _ in range(2):
        xs = [torch.zeros_like(b) for b in bs]
        infos = sem.pcg_solve_batched(ctxs, bs, xs, [1.0] * 4, h2, tol=1e-10, inner=inner)
        assert all(i["status"] == 0 for i in infos), infos
        for c, b, x, h in zip(ctxs, bs, xs, h2):
            alone = torch.zeros_like(b)
            assert c.pcg_solve(b, alone, 1.0, h, tol=1e-10, inner=inner)["status"] == 0
            assert rel(x.cpu().numpy(), alone.cpu().numpy()) <= 1e-9


@pytest.mark.parametrize("restart", [1, 7, 8, 9, 20])
def test_gram_schmidt_group_edges(sem, restart):
    """Krylov bases around the eight vectors that one group of inner products takes."""
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, 4, (3, 4, 3), 0.1)
    bg, bo = fourier_rhs(ctx, m)
    H = sem.HSMG(ctx, [4, 2, 1], dtype="f64")
    x = torch.zeros_like(bg)
    info = H.gmres(bg, x, restart=restart, tol=1e-9, maxit=400)
    assert info["status"] == 0, info
    r, bn = m.residual(bo, x.cpu().numpy(), 1.0, 0.0)
    assert r <= 1.5e-9 * bn
    H.close()


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_replayed_steps_equal_direct_steps(sem, storage):
    """Nine steps on a stream of their own (captured and replayed, one graph per
    arrangement of the history buffers) and on the default stream (launched
    directly) give the same bits."""
    torch, dev = torch_dev()
    out = []
    for st in (torch.cuda.Stream(), torch.cuda.default_stream()):
        ctx, _, _ = pair(sem, 5, (3, 4, 3), 0.0, with_oracle=False)
        T = sem.TGV(ctx, 1.0 / 100, 2e-3)
        T.set_policy([{"storage": storage}])
        x, y, z = gpu_coords(ctx)
        u, v, w, p = inputs.tgv_initial(x, y, z, lib=torch)
        T.set(u.contiguous(), v.contiguous(), (w + 0 * x).contiguous(), p.contiguous())
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            d = T.step(9)
        f = [torch.empty_like(u) for _ in range(4)]
        T.get(*f)
        out.append((f, [r["ke"] for r in d]))
        T.close()
    assert out[0][1] == out[1][1]
    assert all(torch.equal(a, b) for a, b in zip(out[0][0], out[1][0]))


@pytest.mark.parametrize("N", [1, 2, 3, 4, 6, 9])
def test_steps_of_every_parity_match_oracle(sem, N):
    """Two Taylor-Green steps, tight tolerances, at the orders whose interpolations
    fold with and without middle points (N+1 and M odd and even): fields within
    1e-8 of the oracle's."""
    import math

    import oracle
    torch, dev = torch_dev()
    nel, nu, dt = (3, 3, 3), 0.02, 5e-3
    ctx, m, v = pair(sem, N, nel, 0.1)
    tight = sem.opts(tol=1e-12, abs_tol=False)
    T = sem.TGV(ctx, nu, dt, vel=tight, pres=tight)
    x, y, z = gpu_coords(ctx)
    u, vv, w, p = inputs.tgv_initial(x, y, z, lib=torch)
    w = 0.3 * torch.sin(x + 2 * y) + 0 * z
    T.set(u.contiguous(), vv.contiguous(), w.contiguous(), p.contiguous())
    d = T.step(2)
    assert all(r["status"] == 0 for r in d), d
    O = oracle.TGV(N, nel, v, (2 * math.pi,) * 3, nu, dt, tol_v=1e-12, tol_p=1e-12, abs_tol=False)
    xo, yo, zo = m.xyz
    uo, vo, wo, po = inputs.tgv_initial(xo, yo, zo)
    O.set(uo, vo, 0.3 * np.sin(xo + 2 * yo) + 0 * zo, po)
    do = O.step(2)
    out = [torch.empty_like(u) for _ in range(4)]
    T.get(*out)
    for a, b in zip(out[:3], O.get()[:3]):
        assert _err(a.cpu().numpy(), b) <= 1e-8
    # (means over the volume: the quadrature's here, the box's in the oracle, which
    # differ by 1.7e-6 at N = 1, where the quadrature does not integrate det J)
    vol = m.B.sum() / (2 * math.pi) ** 3
    assert abs(d[-1]["ke"] * vol - do[-1, 1]) <= 1e-10 * do[-1, 1]
    assert abs(d[-1]["enstrophy"] * vol - do[-1, 2]) <= 1e-9 * do[-1, 2]
    T.close()
