"""The default wait of the FP64 whole-job kernels for small grids outlasts a launch of half a minute on another stream
(their CTAs may be placed one by one as it leaves the SMs, and the first of them wait for the last): polls of the default
times the time of one, which a wait with a short limit shows."""
import os
import re
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")
POLLS = 1 << 16


def default_polls():
    src = os.path.join(os.path.dirname(os.path.abspath(F.__file__)), "csrc", "resident2d.cuh")
    return 1 << int(re.search(r"RESIDENT_WAIT = 1ll << (\d+)", open(src).read()).group(1))


def step(n, tune):
    p = F.make_problem(2, (n, n), 1.0, "periodic", "const", "fp64")
    ws = torch.empty(F.frkc2_workspace_size(p), dtype=torch.uint8, device="cuda")
    F.frkc2_workspace_reset(ws)
    u = torch.ones(n, n, dtype=torch.float64, device="cuda")
    F.frkc2_step(F.frkc2_plan(8), p, 0.05, 1, 0.0, u, ws, tune)
    return ws


def bruss(n, tune):
    p = F.make_bruss_problem((n, n), bc="periodic", precision="fp64")
    ws = torch.empty(F.frkc2_bruss_workspace_size(p), dtype=torch.uint8, device="cuda")
    F.frkc2_workspace_reset(ws)
    v, w = torch.ones(n, n, dtype=torch.float64, device="cuda"), torch.full((n, n), 3.0, dtype=torch.float64, device="cuda")
    F.frkc2_bruss_step(F.frkc2_plan(8), p, 1e-4, 1, 0.0, v, w, ws, tune)
    return ws


@pytest.mark.parametrize("job,n", [(step, 40), (step, 400), (bruss, 64), (bruss, 200)])
def test_default_wait(job, n):
    job(n, F.make_tuning(wait_limit=POLLS))  # (the first launch loads the kernel)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    ws = job(n, F.make_tuning(wait_limit=POLLS, fault_inject=1))
    torch.cuda.synchronize()
    seconds = time.perf_counter() - t0
    assert F.frkc2_workspace_status(ws) == F.ETIMEOUT
    assert seconds / POLLS * default_polls() > 30.0
