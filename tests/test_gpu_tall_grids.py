"""Grids of some million rows on the FP32 routes that cut a grid into regions, whose rows of regions are more than a launch's
grid has along y."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")


@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("nx,ny", [(16, 2_000_000), (16, 1_400_000)])
def test_bruss_fp32(nx, ny, bc):
    """The same bits as one launch a stage, which has no regions."""
    s = 16
    pr = F.make_bruss_problem((nx, ny), dx=1.0 / 200, bc=bc, precision="fp32")
    plan = F.frkc2_plan(s)
    g = torch.Generator(device="cuda").manual_seed(5)
    v0, w0 = (c + 0.2 * torch.rand(ny, nx, generator=g, device="cuda") for c in (1.0, 3.0))
    ws = torch.empty(F.frkc2_bruss_workspace_size(pr), dtype=torch.uint8, device="cuda")
    out = []
    for kernel in (0, 2):
        F.frkc2_workspace_reset(ws)
        v, w = v0.clone(), w0.clone()
        F.frkc2_bruss_step(plan, pr, 0.9 * plan.info()["beta"] / 6500.0, 1, 0.0, v, w, ws, F.make_tuning(kernel=kernel))
        assert F.frkc2_workspace_status(ws) == F.OK
        out.append((v, w))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
def test_fp32_2d(bc):
    """Against the tile pass of one stage a launch, whose tiles are higher.  Tolerance: both round each of the s stages
    to 2^-24 in their own order, amplified by at most some tens."""
    nx, ny, s = 16, 1_500_000, 16
    pr = F.make_problem(2, (nx, ny), 1.0, bc, "const", "fp32")
    plan = F.frkc2_plan(s)
    g = torch.Generator(device="cuda").manual_seed(6)
    u0 = torch.rand(ny, nx, generator=g, device="cuda")
    ws = torch.empty(F.frkc2_workspace_size(pr), dtype=torch.uint8, device="cuda")
    out = []
    for tune in (None, F.make_tuning(k=1, kernel=1)):
        F.frkc2_workspace_reset(ws)
        u = u0.clone()
        F.frkc2_step(plan, pr, 0.9 * plan.info()["beta"] / 8.0, 1, 0.0, u, ws, tune)
        assert F.frkc2_workspace_status(ws) == F.OK
        out.append(u.double())
    assert (out[0] - out[1]).norm() / out[1].norm() < 1e-5
