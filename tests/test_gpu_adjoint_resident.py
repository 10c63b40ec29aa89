"""The FP64 adjoint whose segments before the last run forward in one launch (small 2D grids) against the same gradient
with a single segment, which has none: one to four segments, a short last one, sizes around the units of that launch.
Tolerance: the two forward runs differ by a few roundings a stage (2^-53), amplified by at most some hundreds."""
import numpy as np
import pytest

from oracle import frkc2_oracle as O
from helpers import oracle_problem, rel_err, seeded_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")


@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
@pytest.mark.parametrize("nx,ny,s,nsteps,ckpt", [(5, 8, 6, 4, 1), (33, 21, 16, 5, 2), (97, 130, 32, 4, 1), (200, 200, 16, 7, 3)])
def test_segments_in_one_launch(nx, ny, s, nsteps, ckpt, bc):
    u0, field = seeded_case((ny, nx), bc, "field", 6100 + nx)
    g, _ = seeded_case((ny, nx), bc, "field", 6200 + ny)
    kt = torch.as_tensor(field, device="cuda")
    pr = F.make_problem(2, (nx, ny), 1.0, bc, "field", "fp64", kappa_field=kt)
    plan = F.frkc2_plan(s)
    dt = 0.9 * O.beta(s) / O.rho_bound(oracle_problem(2, bc, "field", 1.0, field))
    out = []
    for c in (ckpt, nsteps):
        ws = torch.empty(F.frkc2_adjoint_workspace_size(plan, pr, nsteps, c), dtype=torch.uint8, device="cuda")
        F.frkc2_workspace_reset(ws)
        a, b = torch.as_tensor(u0, device="cuda"), torch.as_tensor(g, device="cuda")
        du, dk = torch.empty_like(a), torch.empty_like(kt)
        F.frkc2_adjoint(plan, pr, dt, nsteps, c, a, b, du, dk, ws)
        assert F.frkc2_workspace_status(ws) == F.OK
        out.append((du.cpu().numpy(), dk.cpu().numpy()))
    assert all(np.isfinite(x).all() for x in out[0])
    assert rel_err(out[0][0], out[1][0]) < 1e-11 and rel_err(out[0][1], out[1][1]) < 1e-11
