"""2D passes over padded rows: the FP32 regions with a given k (16-, 8- and 4-byte accesses) and the float-pair
regions, at row lengths of every remainder modulo 4, narrower than a vector and than a region, across the
periodic wrap, with the state at every alignment, and with one pass per step, against the FP64 oracle (the
tolerances of the other parity tests)."""
import numpy as np
import pytest

from oracle import frkc2_oracle as O
from helpers import oracle_problem, rel_err, seeded_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")
TOL = {"fp32": 1e-4, "dfloat": 1e-6}


@pytest.mark.parametrize("prec", ["fp32", "dfloat"])
@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
@pytest.mark.parametrize("nx", [1, 3, 5, 8, 33, 47, 50, 64, 97, 130, 199])
def test_rows_of_every_remainder(nx, bc, prec):
    for ny, s, k, nsteps, offset in [(21, 8, 4, 2, 0), (19, 12, 6, 1, 1), (60, 8, 8, 3, 0), (37, 10, 5, 2, 1)]:
        shape = (ny, nx)
        u0, field = seeded_case(shape, bc, "field", 5100 + nx + ny)
        field = field.astype(np.float32).astype(np.float64)
        u0 = u0.astype(np.float32).astype(np.float64) if prec == "fp32" else u0
        opr = oracle_problem(2, bc, "field", 1.0, field)
        dt = 0.9 * O.beta(s) / O.rho_bound(opr)
        ref = O.frkc2_step(u0, O.plan(s, method="lebedev")["a"], dt, opr, nsteps)
        sd = torch.float32 if prec == "fp32" else torch.float64
        kt = torch.as_tensor(field, dtype=torch.float32, device="cuda")
        pr = F.make_problem(2, (nx, ny), 1.0, bc, "field", prec, kappa_field=kt)
        tune = F.make_tuning(k=k, kernel=3)
        ws = torch.empty(F.frkc2_workspace_size(pr, tune), dtype=torch.uint8, device="cuda")
        F.frkc2_workspace_reset(ws)
        u = torch.empty(ny * nx + 4, dtype=sd, device="cuda")[offset:offset + ny * nx].view(ny, nx)
        u.copy_(torch.as_tensor(u0))
        F.frkc2_step(F.frkc2_plan(s, flags=F.PLAN_LEBEDEV), pr, dt, nsteps, 0.0, u, ws, tune)
        assert F.frkc2_workspace_status(ws) == F.OK
        assert rel_err(u.double().cpu().numpy(), ref) < TOL[prec], (ny, s, k)
