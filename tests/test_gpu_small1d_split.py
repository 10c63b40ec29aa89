"""The 1D whole-job kernel in FP64 with a cell's components on separate lanes (the library's own shape) against the
form with both on one lane (an explicit cluster size, halo period or thread count), bit for bit: sizes at the edges
of a warp's 15 slots, of one warp, of 1 to 8 CTAs of unequal chunks, and of 1, 2, 4 and 8 cells per lane."""
import numpy as np
import pytest

from oracle import frkc2_oracle as O
from helpers import oracle_problem, seeded_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")


@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
@pytest.mark.parametrize("n", [1, 2, 7, 14, 15, 16, 29, 31, 33, 45, 61, 63, 64, 95, 104, 121, 225, 255, 256, 257, 431,
                               511, 700, 833, 976, 4064, 4065, 4097, 7500, 7711, 8200, 15200, 15390, 16384])
def test_split_lanes_same_bits(n, bc):
    u0, field = seeded_case((n,), bc, "field", 8800 + n)
    kt = torch.as_tensor(field, device="cuda")
    pr = F.make_problem(1, (n,), 1.0, bc, "field", "fp64", kappa_field=kt)
    cl = max(1, min(8, n // 32), -(-n // 2048))
    rho = O.rho_bound(oracle_problem(1, bc, "field", 1.0, field), u0)
    for s, nsteps in [(6, 1), (12, 4), (42, 2)]:
        out = []
        for tune in (F.make_tuning(kernel=6), F.make_tuning(kernel=6, tile=(cl, 0, 0))):
            ws = torch.empty(F.frkc2_workspace_size(pr, tune), dtype=torch.uint8, device="cuda")
            F.frkc2_workspace_reset(ws)
            u = torch.as_tensor(u0, device="cuda").clone()
            F.frkc2_step(F.frkc2_plan(s), pr, 0.9 * O.beta(s) / max(rho, 1.0), nsteps, 0.0, u, ws, tune)
            assert F.frkc2_workspace_status(ws) == F.OK
            out.append(u.cpu().numpy())
        assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1]), (n, s)
