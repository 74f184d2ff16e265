"""The CFL number of a step, which makes the next step of a CFL-controlled run, in
FP64: a constant velocity c along x on elements of edge 2 (dr/dx = 1) has U = c
exactly, and the smallest GLL gap is the first node's coordinate, so the number
is dt times c over the gap, each operation rounded once."""
import numpy as np
import pytest

from helpers import gpu_coords, pair, torch_dev

pytestmark = pytest.mark.gpu

C, DT = 0.8125, 0.0078125  # exact in any precision


def _run(sem, N, poison):
    torch, dev = torch_dev()
    nel = (3, 2, 2)
    ctx, _, _ = pair(sem, N, nel, 0.0, L=tuple(2.0 * e for e in nel), with_oracle=False)
    x, _, _ = gpu_coords(ctx)
    T = sem.TGV(ctx, 0.01, DT)
    u, z = torch.full_like(x, C), torch.zeros_like(x)
    if poison:
        u[(N + 1) ** 3 + 5] = float("nan")  # one copy of one node of the second element
    T.set(u, z, z, z)
    d = T.step(1)[0]
    T.close()
    return float(x[1]), d


@pytest.mark.parametrize("N", range(2, 10))
def test_cfl_of_a_constant_velocity(sem, N):
    gap, d = _run(sem, N, False)
    assert d["status"] == 0
    want = C * (1.0 / gap) * DT
    assert abs(d["cfl"] - want) <= 2 * np.spacing(want), (d["cfl"], want)


@pytest.mark.parametrize("N", [4, 7])
def test_cfl_passes_over_a_node_that_is_not_a_number(sem, N):
    gap, d = _run(sem, N, True)
    want = C * (1.0 / gap) * DT
    assert 0.0 <= d["cfl"] <= 100 * want, d
