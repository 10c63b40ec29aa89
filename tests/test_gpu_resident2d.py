"""The FP64 2D whole-job kernel for small grids (the default route there) against the FP64 oracle, at the tolerance of
the other FP64 parity tests: one CTA, units of every width and row count, one unit across a periodic axis, the largest
grids that fit and the first that do not, a captured call, a non-finite state and a wait that runs out."""
import numpy as np
import pytest

from oracle import frkc2_oracle as O
from helpers import oracle_problem, rel_err, seeded_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")
TOL = 1e-11


def setup(nx, ny, bc, kappa="field"):
    u0, field = seeded_case((ny, nx), bc, kappa, 900 + nx + 3 * ny)
    kt = torch.as_tensor(field, device="cuda") if kappa == "field" else None
    pr = F.make_problem(2, (nx, ny), 1.0, bc, kappa, "fp64", kappa_field=kt)
    ws = torch.empty(F.frkc2_workspace_size(pr), dtype=torch.uint8, device="cuda")
    F.frkc2_workspace_reset(ws)
    opr = oracle_problem(2, bc, kappa, 1.0, field)
    return u0, pr, ws, opr, O.rho_bound(opr, u0)


SIZES = [(2, 3, False), (4, 4, False), (5, 8, True), (15, 16, True), (16, 17, True), (17, 33, True), (33, 21, True),
         (31, 64, True), (64, 31, True), (100, 12, True), (7, 300, True), (97, 130, True), (256, 40, True),
         (300, 300, True), (512, 512, True), (2432, 8, True), (2433, 8, True), (600, 600, False)]


@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
@pytest.mark.parametrize("nx,ny,resident", SIZES)
def test_whole_job(nx, ny, resident, bc):
    for s, nsteps, kappa in [(6, 1, "field"), (16, 3, "const")]:
        u0, pr, ws, opr, rho = setup(nx, ny, bc, kappa)
        dt = 0.9 * O.beta(s) / max(rho, 1e-3)
        ref = O.frkc2_step(u0, O.plan(s)["a"], dt, opr, nsteps)
        u = torch.as_tensor(u0, device="cuda").clone()
        F.frkc2_launch_count()
        F.frkc2_step(F.frkc2_plan(s), pr, dt, nsteps, 0.0, u, ws)
        if torch.cuda.get_device_properties(0).multi_processor_count == 152:
            assert F.frkc2_launch_count() == (2 if resident else 2 + s * nsteps)
        assert F.frkc2_workspace_status(ws) == F.OK
        assert rel_err(u.cpu().numpy(), ref) < TOL


def test_captured_and_repeated():
    """A captured call replayed: the packets of one run are not taken for the next one's."""
    s = 12
    u0, pr, ws, opr, rho = setup(77, 54, "periodic")
    dt = 0.9 * O.beta(s) / rho
    plan, u = F.frkc2_plan(s), torch.as_tensor(u0, device="cuda").clone()
    F.frkc2_step(plan, pr, dt, 2, 0.0, u, ws)
    u.copy_(torch.as_tensor(u0))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        F.frkc2_step(plan, pr, dt, 2, 0.0, u, ws)
    u.copy_(torch.as_tensor(u0))
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert F.frkc2_workspace_status(ws) == F.OK
    assert rel_err(u.cpu().numpy(), O.frkc2_step(u0, O.plan(s)["a"], dt, opr, 6)) < TOL


def test_two_streams():
    """Whole jobs on two streams at a time, each of a size that fills the SMs' registers: each ends as it does alone."""
    s, jobs = 16, []
    for nx, ny in [(512, 512), (384, 400)]:
        u0, pr, ws, opr, rho = setup(nx, ny, "periodic")
        jobs.append((F.frkc2_plan(s), pr, 0.9 * O.beta(s) / rho, torch.as_tensor(u0, device="cuda"), ws, torch.cuda.Stream()))
    out = []
    for together in (False, True):
        got = []
        for plan, pr, dt, u0, ws, st in jobs:
            u = u0.clone()
            torch.cuda.synchronize()
            got.append((u, ws))
        for rep in range(5):
            for (plan, pr, dt, u0, ws, st), (u, _) in zip(jobs, got):
                with torch.cuda.stream(st):
                    F.frkc2_step(plan, pr, dt, 3, 0.0, u, ws)
                if not together:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert all(F.frkc2_workspace_status(ws) == F.OK for _, ws in got)
        out.append([u.cpu().numpy() for u, _ in got])
    assert all(np.array_equal(a, b) for a, b in zip(*out))


def test_beside_a_persistent_launch():
    """A whole job queued while a persistent batched launch holds the SMs' registers on another stream: both end as alone."""
    s, n = 64, 600
    plan = F.frkc2_plan(s)
    probs, us, dts = [], [], []
    for i in range(6):
        u0, field = seeded_case((n, n), "periodic", "field", 70 + i)
        kt = torch.as_tensor(field, device="cuda")
        probs.append(F.make_problem(2, (n, n), 1.0, "periodic", "field", "fp64", kappa_field=kt))
        us.append(torch.as_tensor(u0, device="cuda"))
        dts.append(0.9 * O.beta(s) / O.rho_bound(oracle_problem(2, "periodic", "field", 1.0, field)))
    steps, plans = [4] * 6, [plan] * 6
    u0, pr, ws, opr, rho = setup(512, 500, "periodic")
    dt, side = 0.9 * O.beta(s) / rho, torch.cuda.Stream()
    out = []
    for together in (False, True):
        bu, u = [t.clone() for t in us], torch.as_tensor(u0, device="cuda").clone()
        bws = torch.empty(F.frkc2_batch_workspace_size(plans, probs, steps), dtype=torch.uint8, device="cuda")
        F.frkc2_workspace_reset(bws)
        F.frkc2_batch_prepare(plans, probs, dts, steps, bu, bws)
        torch.cuda.synchronize()
        F.frkc2_batch_launch(bws)
        if not together:
            torch.cuda.synchronize()
        with torch.cuda.stream(side):
            F.frkc2_step(plan, pr, dt, 3, 0.0, u, ws)
        torch.cuda.synchronize()
        assert F.frkc2_workspace_status(ws) == F.OK and F.frkc2_workspace_status(bws) == F.OK
        out.append([t.cpu().numpy() for t in bu + [u]])
    assert all(np.array_equal(a, b) for a, b in zip(*out))


def test_status():
    s = 8
    u0, pr, ws, opr, rho = setup(60, 50, "dirichlet")
    dt = 0.9 * O.beta(s) / rho
    plan, u = F.frkc2_plan(s), torch.as_tensor(u0, device="cuda").clone()
    F.frkc2_step(plan, pr, dt, 1, 0.0, u, ws, F.make_tuning(wait_limit=1000, fault_inject=1))
    assert F.frkc2_workspace_status(ws) == F.ETIMEOUT
    F.frkc2_workspace_reset(ws)
    u.copy_(torch.as_tensor(u0))
    F.frkc2_step(plan, pr, dt, 1, 0.0, u, ws)
    assert F.frkc2_workspace_status(ws) == F.OK
    assert rel_err(u.cpu().numpy(), O.frkc2_step(u0, O.plan(s)["a"], dt, opr, 1)) < TOL
    u[3, 4] = float("nan")
    F.frkc2_step(plan, pr, dt, 1, 0.0, u, ws)
    assert F.frkc2_workspace_status(ws) == F.ENONFINITE
