"""Solves whose bounded wait runs out (a limit far below the time of one grid
barrier; nothing hangs): what they leave on the context must not reach later
solves.  The mesh is deformed and the problems Helmholtz, so that a diagonal
that was not assembled or inverted changes the iterations.  The later solve does
the same arithmetic as on a context of its own: the same bits.
"""
import pytest

from helpers import fourier_rhs, gpu_coords, pair, torch_dev
from paper_2608_24348_gb300 import inputs

pytestmark = pytest.mark.gpu

LIMIT = 1e-9  # seconds


@pytest.mark.parametrize("inner", ["f64", "f32", "f64_native"])
@pytest.mark.parametrize("info", [True, False])
@pytest.mark.parametrize("N", [6, 7])
def test_later_solve_makes_its_own_preconditioner(sem, inner, info, N):
    torch, dev = torch_dev()
    out = []
    for interrupted in (False, True):
        ctx, m, _ = pair(sem, N, (3, 4, 3), 0.1, with_oracle=False)
        bg, _ = fourier_rhs(ctx, m)
        x = torch.zeros_like(bg)
        if interrupted:
            ctx.pcg_solve(bg, x, 1.0, 3.0, inner=inner, wait_timeout_s=LIMIT, sync=info)
            torch.cuda.synchronize()
            assert ctx.last_solve_info()["status"] == sem.ERR_TIMEOUT
            x.zero_()
        d = ctx.pcg_solve(bg, x, 1.0, 3.0, tol=1e-10, inner=inner)
        assert d["status"] == 0, d
        out.append((d["iters"], x))
    assert out[0][0] == out[1][0]
    assert torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("inner", ["f64", "f64_native"])
def test_residual_norm_of_an_interrupted_solve(sem, inner):
    """The limit is halved between one that stops the solve at once and one that
    does not stop it, until a solve stops on its way; the norm it reports is that of
    a solve of as many iterations."""
    torch, dev = torch_dev()
    ctx, m, _ = pair(sem, 7, (9, 8, 7), 0.1, with_oracle=False)
    bg, _ = fourier_rhs(ctx, m)
    x = torch.zeros_like(bg)
    lo, hi, info = 1e-9, 1e-3, None
    for _ in range(60):
        limit = (lo * hi) ** 0.5
        x.zero_()
        d = ctx.pcg_solve(bg, x, 1.0, 0.0, tol=1e-10, inner=inner, wait_timeout_s=limit)
        if d["status"] != sem.ERR_TIMEOUT:
            hi = limit
        elif d["iters"] == 0:
            lo = limit
        else:
            info = d
            break
    if info is None:
        pytest.skip("no limit stopped the solve on its way")
    x.zero_()
    ref = ctx.pcg_solve(bg, x, 1.0, 0.0, tol=1e-10, inner=inner, maxit=info["iters"])
    assert ref["iters"] == info["iters"]
    assert abs(info["rnorm"] - ref["rnorm"]) <= 1e-9 * ref["rnorm"], (info, ref)


@pytest.mark.parametrize("inner", ["f64", "f32"])
@pytest.mark.parametrize("orders", [(7, 5), (7, 4)])  # one launch; a launch for each problem
def test_later_batch_makes_its_own_preconditioners(sem, inner, orders):
    torch, dev = torch_dev()
    out = []
    for interrupted in (False, True):
        a, _, _ = pair(sem, orders[0], (3, 2, 3), 0.1, with_oracle=False)
        c, _, _ = pair(sem, orders[1], (4, 3, 3), 0.1, with_oracle=False)
        ctxs = [a, c, a, a]
        bs = [fourier_rhs(t, None)[0] for t in ctxs]
        xs = [torch.zeros_like(b) for b in bs]
        if interrupted:
            infos = sem.pcg_solve_batched(ctxs, bs, xs, [1.0] * 4, [4.0, 1.0, 4.0, 9.0], inner=inner,
                                          wait_timeout_s=LIMIT)
            assert all(i["status"] == sem.ERR_TIMEOUT for i in infos), infos
            for x in xs:
                x.zero_()
        infos = sem.pcg_solve_batched(ctxs, bs, xs, [1.0] * 4, [4.0, 1.0, 4.0, 9.0], inner=inner, tol=1e-10)
        assert all(i["status"] == 0 for i in infos), infos
        out.append(([i["iters"] for i in infos], xs))
    assert out[0][0] == out[1][0]
    assert all(torch.equal(p, q) for p, q in zip(out[0][1], out[1][1]))


def test_later_stepper_makes_its_own_preconditioners(sem):
    """Two steppers on one context use the same solver workspaces."""
    torch, dev = torch_dev()
    out = []
    for interrupted in (False, True):
        ctx, _, _ = pair(sem, 5, (3, 4, 3), 0.1, with_oracle=False)
        x, y, z = gpu_coords(ctx)
        f = [(t + 0 * x).contiguous() for t in inputs.tgv_initial(x, y, z, lib=torch)]
        if interrupted:
            o = sem.opts(tol=1e-8, wait_timeout_s=LIMIT)
            T = sem.TGV(ctx, 0.02, 5e-3, vel=o, pres=o)
            T.set(*f)
            assert T.step(1)[0]["status"] == sem.ERR_TIMEOUT
            T.close()
        o = sem.opts(tol=1e-8)
        T = sem.TGV(ctx, 0.02, 5e-3, vel=o, pres=o)
        T.set(*f)
        d = T.step(2)
        assert all(r["status"] == 0 for r in d), d
        g = [torch.empty_like(x) for _ in range(4)]
        T.get(*g)
        T.close()
        out.append(([r["iters"] for r in d], g))
    assert out[0][0] == out[1][0]
    assert all(torch.equal(p, q) for p, q in zip(out[0][1], out[1][1]))
