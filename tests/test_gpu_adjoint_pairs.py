"""The FP32 adjoint's tape and reverse passes with pair access (even rows) and without (odd rows), and the stage
counts they choose per pass, against the FP64 adjoint of the same problem: sizes around the regions' tiles, one
and several segments, stage counts that leave a short last pass.  Tolerance: the float rounding of the state,
2^-24, through the rounding gain of the stage order and of its reverse (some hundreds at s = 32), below 1e-3."""
import pytest

from helpers import rel_err, seeded_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")


def gradients(prec, shape, bc, s, nsteps, ckpt, u0, field, g, dt):
    sd = torch.float64 if prec == "fp64" else torch.float32
    kt = torch.as_tensor(field, dtype=sd, device="cuda")
    pr = F.make_problem(2, tuple(reversed(shape)), 1.0, bc, "field", prec, kappa_field=kt)
    plan = F.frkc2_plan(s, flags=F.PLAN_LEBEDEV)
    ws = torch.empty(F.frkc2_adjoint_workspace_size(plan, pr, nsteps, ckpt), dtype=torch.uint8, device="cuda")
    F.frkc2_workspace_reset(ws)
    a, b = (torch.as_tensor(x, dtype=sd, device="cuda") for x in (u0, g))
    du, dk = torch.empty_like(a), torch.empty_like(kt)
    F.frkc2_adjoint(plan, pr, dt, nsteps, ckpt, a, b, du, dk, ws)
    assert F.frkc2_workspace_status(ws) == F.OK
    return du.double().cpu().numpy(), dk.double().cpu().numpy()


@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
@pytest.mark.parametrize("shape,s,nsteps,ckpt", [((3, 4), 4, 2, 1), ((40, 40), 22, 2, 2), ((41, 43), 22, 2, 2), ((65, 80), 32, 3, 2),
                                                 ((200, 402), 10, 1, 1), ((611, 700), 16, 1, 1), ((611, 701), 16, 1, 1)])
def test_fp32_adjoint_passes_match_fp64(shape, s, nsteps, ckpt, bc):
    u0, field = seeded_case(shape, bc, "field", 4100 + sum(shape))
    g, _ = seeded_case(shape, bc, "field", 4200 + sum(shape))
    dt = 0.9 * 2.0 * (s * s - 1) / 3.0 / (8.0 * field.max())
    ref = gradients("fp64", shape, bc, s, nsteps, ckpt, u0, field, g, dt)
    got = gradients("fp32", shape, bc, s, nsteps, ckpt, u0, field, g, dt)
    assert rel_err(got[0], ref[0]) < 1e-3 and rel_err(got[1], ref[1]) < 1e-3
