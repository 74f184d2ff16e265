"""The stepper's history levels where their buffers turn, are written in place or
are taken by a graph of the caller's: what a step leaves in them has to be what
the same steps alone leave, bit for bit."""
import pytest

from helpers import gpu_coords, pair, torch_dev
from paper_2608_24348_gb300 import inputs

pytestmark = pytest.mark.gpu


def _stepper(sem, N=5, nel=(3, 4, 3), **kw):
    """A stepper in the middle of a run: three different velocity levels."""
    torch, dev = torch_dev()
    ctx, _, _ = pair(sem, N, nel, 0.05, with_oracle=False)
    T = sem.TGV(ctx, 0.02, 4e-3, **kw)
    x, y, z = gpu_coords(ctx)
    u, v, w, p = (t + 0 * x for t in inputs.tgv_initial(x, y, z, lib=torch))
    w = w + 0.2 * torch.sin(x + 2 * y)
    for level in (2, 1, 0):
        s = 1.0 + 0.01 * level
        T.set(s * u, s * v, s * w, p.contiguous() if level == 0 else None, level=level, step=3)
    return ctx, T


def _state(T, ctx):
    torch, dev = torch_dev()
    f = [torch.empty(ctx.nL, dtype=torch.float64, device=dev) for _ in range(4)]
    T.get(*f)
    return f


def _same(a, b):
    torch, _ = torch_dev()
    return all(torch.equal(p, q) for p, q in zip(a, b))


@pytest.mark.parametrize("which", ["vel", "pres"])
def test_a_refused_step_leaves_the_state(sem, which):
    """The split-operand inner operators end at N = 7: a step with them at N = 8 is
    refused; after a policy that asks for FP64 solves the run goes on as if it had
    not been tried."""
    opts = {which: sem.opts(tol=1e-8, inner="f16x2_tc")}
    other = "pres" if which == "vel" else "vel"
    opts[other] = sem.opts(tol=1e-8)
    out = []
    for tried in (False, True):
        ctx, T = _stepper(sem, 8, (3, 2, 3), **opts)
        if tried:
            before = _state(T, ctx)
            with pytest.raises(sem.SemError):
                T.step(1)
            assert _same(before, _state(T, ctx))
        T.set_policy([{}])
        d = T.step(3)
        assert all(r["status"] == 0 for r in d), d
        out.append(_state(T, ctx))
        T.close()
    assert _same(*out)


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("direct", [4, 5])
def test_replays_of_a_step_captured_by_the_caller(sem, storage, direct):
    """One captured step replayed five times is five steps, from either arrangement
    of the history buffers, and the stepper goes on from there."""
    torch, dev = torch_dev()
    out = []
    for captured in (False, True):
        ctx, T = _stepper(sem, vel=sem.opts(tol=1e-8), pres=sem.opts(tol=1e-8))
        T.set_policy([{"storage": storage}])
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        T.step(direct, diag=False, stream=st)
        if captured:
            st.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st):
                T.step(1, diag=False, stream=st)
            for _ in range(5):
                g.replay()
            torch.cuda.synchronize()
        else:
            T.step(5, diag=False, stream=st)
        T.step(2, diag=False, stream=st)
        torch.cuda.synchronize()
        out.append(_state(T, ctx))
        T.close()
    assert _same(*out)


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("direct", [1, 2, 3])
def test_levels_set_between_steps(sem, storage, direct):
    """The levels that sem_tgv_set writes are those the next steps read, from every
    arrangement of the history buffers."""
    torch, dev = torch_dev()
    out = []
    for before in (0, direct):
        ctx, T = _stepper(sem, vel=sem.opts(tol=1e-8), pres=sem.opts(tol=1e-8))
        T.set_policy([{"storage": storage}])
        T.step(3)  # (the storage is the policy's from the first step on)
        T.step(before)
        x, y, z = gpu_coords(ctx)
        u, v, w, p = (t + 0 * x for t in inputs.tgv_initial(x, y, z, lib=torch))
        for level in (2, 1, 0):
            s = 0.9 + 0.02 * level
            T.set(s * u, s * v, w.contiguous(), p.contiguous() if level == 0 else None, level=level, step=3)
        T.step(3)
        out.append(_state(T, ctx))
        T.close()
    assert _same(*out)


def test_a_stepper_takes_no_more_memory_than_its_fields(sem):
    """32 FP64 E-vectors of fields and workspace are enough for a step (29 of the
    stepper and two of the mass); with J^-1 (9 + 4.5 on the context, 9 as pairs) and
    four solver workspaces (7.5 each).  An E-vector here is 16 MiB."""
    torch, dev = torch_dev()
    ctx, _, _ = pair(sem, 7, (16, 16, 16), 0.0, with_oracle=False)
    vec = 8 * ctx.nL
    assert vec == 16 << 20
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    T = sem.TGV(ctx, 0.02, 1e-3)
    used = before - torch.cuda.mem_get_info()[0]
    T.close()
    assert used <= (32 + 22.5 + 30) * vec + (8 << 20), used / vec
