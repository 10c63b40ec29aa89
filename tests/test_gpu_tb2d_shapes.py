"""The FP32 2D pass with the library's choice of region size and stages per pass: grids that take 32 x 32 and
64 x 64 regions, sizes around the tiles' edges, stage counts that leave short last passes, and one pass per
step, against the FP64 oracle (the tolerance of the other FP32 parity tests)."""
import numpy as np
import pytest

from oracle import frkc2_oracle as O
from helpers import oracle_problem, rel_err, seeded_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")


@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
@pytest.mark.parametrize("shape,s,nsteps", [((1, 1), 2, 3), ((3, 5), 4, 2), ((12, 13), 10, 2), ((16, 48), 8, 1), ((32, 33), 22, 2),
                                            ((61, 129), 16, 2), ((200, 131), 32, 1), ((257, 255), 16, 2), ((401, 399), 16, 1),
                                            ((610, 701), 12, 1), ((777, 1021), 8, 1)])
def test_chosen_regions_match_oracle(shape, s, nsteps, bc):
    u0, field = seeded_case(shape, bc, "field", 3100 + sum(shape))
    u0 = u0.astype(np.float32).astype(np.float64)
    field = field.astype(np.float32).astype(np.float64)
    opr = oracle_problem(2, bc, "field", 1.0, field)
    dt = 0.9 * O.beta(s) / O.rho_bound(opr)
    ref = O.frkc2_step(u0, O.plan(s, method="lebedev")["a"], dt, opr, nsteps)
    kt = torch.as_tensor(field, dtype=torch.float32, device="cuda")
    pr = F.make_problem(2, tuple(reversed(shape)), 1.0, bc, "field", "fp32", kappa_field=kt)
    ws = torch.empty(F.frkc2_workspace_size(pr), dtype=torch.uint8, device="cuda")
    F.frkc2_workspace_reset(ws)
    u = torch.as_tensor(u0, dtype=torch.float32, device="cuda")
    F.frkc2_step(F.frkc2_plan(s, flags=F.PLAN_LEBEDEV), pr, dt, nsteps, 0.0, u, ws)
    assert F.frkc2_workspace_status(ws) == F.OK
    assert rel_err(u.double().cpu().numpy(), ref) < 1e-4
