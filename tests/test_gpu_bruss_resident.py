"""The Brusselator's FP64 whole-job kernel for small grids (the default route there) against the oracle, at the tolerance
of the other FP64 parity tests: units of every width and row count, one unit across an axis, both boundary conditions, the
largest grids that fit and grids that keep the persistent kernel, a captured call, a non-finite state and a wait that runs out."""
import numpy as np
import pytest

from oracle import brusselator as BR
from oracle import frkc2_oracle as O
from helpers import rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")
TOL = 1e-11


def setup(nx, ny, bc):
    r = np.random.default_rng(31 * nx + ny)
    v0, w0 = 1.0 + 0.2 * r.standard_normal((ny, nx)), 3.0 + 0.2 * r.standard_normal((ny, nx))
    pr = BR.problem((ny, nx), bc=bc)
    p = F.make_bruss_problem((nx, ny), bc=bc, precision="fp64")
    ws = torch.empty(F.frkc2_bruss_workspace_size(p), dtype=torch.uint8, device="cuda")
    F.frkc2_workspace_reset(ws)
    return v0, w0, pr, p, ws, BR.rho_bound(v0, w0, pr)


def state(v0, w0):
    return torch.as_tensor(v0, device="cuda").clone(), torch.as_tensor(w0, device="cuda").clone()


@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 9), (9, 1), (2, 3), (16, 4), (15, 16), (17, 33), (31, 20), (33, 21), (64, 64),
                                   (130, 97), (7, 300), (300, 7), (200, 200), (256, 256), (400, 400), (500, 512), (610, 600),
                                   (34, 411), (457, 355), (247, 777), (619, 305), (420, 269)])
def test_whole_job(nx, ny, bc):
    v0, w0, pr, p, ws, rho = setup(nx, ny, bc)
    for s, nsteps in [(6, 1), (16, 2)]:
        dt = min(0.8 * O.beta(s) / rho, 0.05)  # (beyond, the reaction of the smallest grids overflows in the oracle too)
        rv, rw = BR.frkc2_step(v0, w0, O.plan(s)["a"], dt, pr, nsteps)
        v, w = state(v0, w0)
        F.frkc2_bruss_step(F.frkc2_plan(s), p, dt, nsteps, 0.0, v, w, ws)
        assert F.frkc2_workspace_status(ws) == F.OK
        assert rel_err(v.cpu().numpy(), rv) < TOL and rel_err(w.cpu().numpy(), rw) < TOL


def test_captured_and_repeated():
    s = 12
    v0, w0, pr, p, ws, rho = setup(77, 54, "periodic")
    dt, plan = min(0.5 * O.beta(s) / rho, 0.05), F.frkc2_plan(s)
    v, w = state(v0, w0)
    F.frkc2_bruss_step(plan, p, dt, 2, 0.0, v, w, ws)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        F.frkc2_bruss_step(plan, p, dt, 2, 0.0, v, w, ws)
    v.copy_(torch.as_tensor(v0))
    w.copy_(torch.as_tensor(w0))
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert F.frkc2_workspace_status(ws) == F.OK
    rv, rw = BR.frkc2_step(v0, w0, O.plan(s)["a"], dt, pr, 6)
    assert rel_err(v.cpu().numpy(), rv) < TOL and rel_err(w.cpu().numpy(), rw) < TOL


def test_status():
    s = 8
    v0, w0, pr, p, ws, rho = setup(60, 50, "neumann")
    dt, plan = min(0.5 * O.beta(s) / rho, 0.05), F.frkc2_plan(s)
    v, w = state(v0, w0)
    F.frkc2_bruss_step(plan, p, dt, 1, 0.0, v, w, ws, F.make_tuning(wait_limit=1000, fault_inject=1))
    assert F.frkc2_workspace_status(ws) == F.ETIMEOUT
    F.frkc2_workspace_reset(ws)
    v, w = state(v0, w0)
    F.frkc2_bruss_step(plan, p, dt, 1, 0.0, v, w, ws)
    assert F.frkc2_workspace_status(ws) == F.OK
    rv, rw = BR.frkc2_step(v0, w0, O.plan(s)["a"], dt, pr, 1)
    assert rel_err(v.cpu().numpy(), rv) < TOL and rel_err(w.cpu().numpy(), rw) < TOL
    w[3, 4] = float("inf")
    F.frkc2_bruss_step(plan, p, dt, 1, 0.0, v, w, ws)
    assert F.frkc2_workspace_status(ws) == F.ENONFINITE
