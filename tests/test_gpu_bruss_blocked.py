"""The temporally blocked FP32 Brusselator passes (the FP32 default) against one launch per stage: the same
bits, at sizes around the regions' edges (32 and 64 cells less the halo), smaller than a region, unaligned
rows (scalar loads), both boundary kinds, and stage counts that leave a short last pass."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")


def run(shape, bc, s, nsteps, kernel, offset=0):
    ny, nx = shape
    rng = np.random.default_rng(nx * 1000 + ny)
    pr = F.make_bruss_problem((nx, ny), dx=1.0 / 200, bc=bc, precision="fp32")
    plan = F.frkc2_plan(s)
    dt = 0.9 * plan.info()["beta"] / 6500.0
    ws = torch.empty(F.frkc2_bruss_workspace_size(pr), dtype=torch.uint8, device="cuda")
    F.frkc2_workspace_reset(ws)
    base = [torch.empty(ny * nx + 4, dtype=torch.float32, device="cuda") for _ in range(2)]
    v, w = (b[offset:offset + ny * nx].view(ny, nx) for b in base)
    v.copy_(torch.as_tensor(1.0 + 0.2 * rng.uniform(-1, 1, shape)))
    w.copy_(torch.as_tensor(3.0 + 0.2 * rng.uniform(-1, 1, shape)))
    F.frkc2_bruss_step(plan, pr, dt, nsteps, 0.0, v, w, ws, F.make_tuning(kernel=kernel))
    return v.cpu(), w.cpu(), F.frkc2_workspace_status(ws)


@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("shape,s", [((1, 1), 2), ((3, 2), 4), ((20, 24), 16), ((16, 17), 8), ((33, 96), 10), ((144, 144), 16),
                                     ((201, 200), 16), ((611, 700), 12), ((900, 1100), 8), ((1030, 2048), 16)])
def test_blocked_passes_equal_per_stage_launches(shape, s, bc):
    a = run(shape, bc, s, 2, 0)
    b = run(shape, bc, s, 2, 2)
    assert a[2] == F.OK and b[2] == F.OK
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


def test_unaligned_state_and_nonfinite():
    a = run((48, 96), "periodic", 8, 1, 0, offset=1)
    b = run((48, 96), "periodic", 8, 1, 2, offset=0)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    pr = F.make_bruss_problem((96, 48), dx=1.0 / 200, bc="neumann", precision="fp32")
    ws = torch.empty(F.frkc2_bruss_workspace_size(pr), dtype=torch.uint8, device="cuda")
    F.frkc2_workspace_reset(ws)
    v = torch.ones(48, 96, device="cuda")
    w = torch.full((48, 96), 3.0, device="cuda")
    v[47, 95] = float("nan")
    F.frkc2_bruss_step(F.frkc2_plan(8), pr, 1e-5, 1, 0.0, v, w, ws)
    assert F.frkc2_workspace_status(ws) == F.ENONFINITE
