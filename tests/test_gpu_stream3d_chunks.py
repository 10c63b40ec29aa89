"""The 3D streaming passes give a cell the same bits wherever along z the chunks of a launch begin: on a periodic box the
state shifted by some planes gives the result shifted by as many.  (MIXED keeps one face of 32 apart, so it is shifted by
multiples of 32.)"""
import pytest

from helpers import seeded_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")


@pytest.mark.parametrize("shape", [(96, 20, 33), (64, 40, 61), (200, 7, 31)])
@pytest.mark.parametrize("prec,kappa,exponent,shifts", [("fp64", "power", 2.5, (1, 5, 33)), ("fp32", "power", 2.5, (1, 5, 33)),
                                                        ("fp64", "power", 1.7, (1, 33)), ("fp64", "field", 2.5, (1, 33)),
                                                        ("fp32", "field", 2.5, (1, 33)), ("mixed", "power", 2.5, (32,))])
def test_shifted_planes(shape, prec, kappa, exponent, shifts):
    if prec == "mixed" and shape[0] % 32:
        pytest.skip("its planes would meet the box's ends elsewhere")
    u0, field = seeded_case(shape, "periodic", kappa, 2900 + sum(shape))
    dtype = torch.float32 if prec == "fp32" else torch.float64
    u0 = torch.as_tensor(u0, dtype=dtype, device="cuda")
    plan, rho = F.frkc2_plan(16), torch.zeros(1, dtype=torch.float64, device="cuda")

    def run(shift):
        kt = None if field is None else torch.as_tensor(field, dtype=dtype, device="cuda").roll(shift, 0).contiguous()
        pr = F.make_problem(3, tuple(reversed(shape)), 1.0, "periodic", kappa, prec, kappa_p=exponent, kappa_field=kt)
        ws = torch.empty(F.frkc2_workspace_size(pr), dtype=torch.uint8, device="cuda")
        F.frkc2_workspace_reset(ws)
        u = u0.roll(shift, 0).contiguous()
        F.frkc2_rho_bound(pr, u, rho)
        F.frkc2_step(plan, pr, 0.9 * plan.info()["beta"] / rho.item(), 2, rho.item(), u, ws)
        assert F.frkc2_workspace_status(ws) == F.OK
        return u.roll(-shift, 0)

    want = run(0)
    for shift in shifts:
        assert torch.equal(run(shift), want), shift
