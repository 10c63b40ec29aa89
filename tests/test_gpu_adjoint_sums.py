"""dJ/dkappa of the FP32 adjoint sums at most 8 stages in FP32 before it widens the sum.  The steps make that visible: 8
large ones, 8 that are 2^-27 of them, 8 large of the other sign.  The large terms cancel and the small remain, unless they
were added to the large in FP32 (in a pass of 10 or 12 stages, say).  The state and lambda stay constant (dt = 2^-50) and
vary along x only, so that the terms of a cell come from its own stage.  Tolerance: the FP64 adjoint's own changes of
state, 2^-50 of terms 2^24 times the result."""
import numpy as np
import pytest

from helpers import rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")


@pytest.mark.parametrize("nx,ny", [(64, 40), (200, 200), (2, 9), (36, 36), (130, 65), (63, 40)])
def test_at_most_eight_stages_in_fp32(nx, ny):
    r = np.random.default_rng(nx)
    plan = F.frkc2_plan_from_steps(np.repeat([-1.0, 2.0 ** -27, 1.0], 8))  # (the adjoint goes from the last)
    u0, g = (np.tile(r.uniform(0.5, 1.0, nx).astype(np.float32), (ny, 1)) for _ in range(2))
    out = []
    for dtype, prec in ((torch.float32, "fp32"), (torch.float64, "fp64")):
        kt = torch.ones(ny, nx, dtype=dtype, device="cuda")
        pr = F.make_problem(2, (nx, ny), 1.0, "periodic", "field", prec, kappa_field=kt)
        ws = torch.empty(F.frkc2_adjoint_workspace_size(plan, pr, 1, 1), dtype=torch.uint8, device="cuda")
        F.frkc2_workspace_reset(ws)
        a, b = (torch.as_tensor(x, dtype=dtype, device="cuda") for x in (u0, g))
        du, dk = torch.empty_like(a), torch.empty_like(kt)
        F.frkc2_adjoint(plan, pr, 2.0 ** -50, 1, 1, a, b, du, dk, ws)
        assert F.frkc2_workspace_status(ws) == F.OK
        out.append(dk.double().cpu().numpy())
    assert np.abs(out[1]).max() > 0
    assert rel_err(out[0], out[1]) < 1e-5
