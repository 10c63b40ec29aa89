"""A 3D FP32 problem whose planes are larger than the packed pass addresses (2^29 cells), against the tile pass.  Tolerance: both
round the s stages to 2^-24 in their own order, amplified by at most some tens."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")


@pytest.mark.parametrize("bc,kappa", [("periodic", "power"), ("dirichlet", "const")])
def test_fp32_plane_above_2_29_cells(bc, kappa):
    nx, ny, s = 4099, 131_001, 4
    pr = F.make_problem(3, (nx, ny, 1), 1.0, bc, kappa, "fp32", kappa_c=0.5)
    plan = F.frkc2_plan(s)
    u0 = torch.rand(1, ny, nx, generator=torch.Generator(device="cuda").manual_seed(7), device="cuda")
    ws = torch.empty(F.frkc2_workspace_size(pr), dtype=torch.uint8, device="cuda")
    out = []
    for tune in (None, F.make_tuning(k=1, kernel=1)):
        F.frkc2_workspace_reset(ws)
        u = u0.clone()
        F.frkc2_step(plan, pr, 0.9 * plan.info()["beta"] / 18.0, 1, 0.0, u, ws, tune)
        assert F.frkc2_workspace_status(ws) == F.OK
        out.append(u)
    diff = sum((a.double() - b.double()).square().sum() for a, b in zip(out[0].split(8192, 1), out[1].split(8192, 1))).sqrt()
    assert diff / out[1].double().norm() < 1e-5
