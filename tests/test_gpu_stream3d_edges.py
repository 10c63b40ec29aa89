"""The 3D streaming passes at the edges of their blocks: columns around multiples of the 30 outputs of a
warp, rows around the outputs of a CTA, one and a few planes, every precision, boundary and conductivity
kind, against the FP64 oracle; and MIXED where its integer conversions do not apply."""
import numpy as np
import pytest

from oracle import frkc2_oracle as O
from helpers import oracle_problem, rel_err, seeded_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = pytest.importorskip("paper_1702_03818_gb300.frkc2")

SDT = {"fp64": torch.float64, "fp32": torch.float32, "mixed": torch.float64}
KDT = {"fp64": torch.float64, "fp32": torch.float32, "mixed": torch.float32}
TOL = {"fp64": 1e-11, "fp32": 1e-4, "mixed": 1e-6}  # those of the other forward parity tests


def run(prob, plan, u0, dt, nsteps, prec, tune=None):
    ws = torch.empty(F.frkc2_workspace_size(prob, tune), dtype=torch.uint8, device="cuda")
    F.frkc2_workspace_reset(ws)
    u = torch.as_tensor(u0, dtype=SDT[prec], device="cuda")
    F.frkc2_step(plan, prob, dt, nsteps, 0.0, u, ws, tune)
    return u.double().cpu().numpy(), F.frkc2_workspace_status(ws)


# shape (z, y, x): 30 output columns a block; output rows 14, 10, 6 (FP32) or 30 .. 14 (double state)
@pytest.mark.parametrize("shape", [(1, 6, 30), (2, 7, 31), (3, 14, 29), (5, 15, 61), (4, 30, 60), (33, 31, 33), (65, 3, 62)])
@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
@pytest.mark.parametrize("kappa", ["field", "power"])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "mixed"])
def test_block_edges_match_oracle(shape, bc, kappa, prec):
    s = 8
    u0, field = seeded_case(shape, bc, kappa, 2100 + sum(shape))
    fo = field if field is None or prec == "fp64" else field.astype(np.float32).astype(np.float64)
    u0o = u0.astype(np.float32).astype(np.float64) if prec == "fp32" else u0
    opr = oracle_problem(3, bc, kappa, 1.0, fo)
    dt = 0.9 * O.beta(s) / O.rho_bound(opr, u0o)
    ref = O.frkc2_step(u0o, O.plan(s)["a"], dt, opr, 2)
    kt = torch.as_tensor(field, dtype=KDT[prec], device="cuda") if field is not None else None
    pr = F.make_problem(3, tuple(reversed(shape)), 1.0, bc, kappa, prec, kappa_field=kt)
    got, st = run(pr, F.frkc2_plan(s), u0, dt, 2, prec, F.make_tuning(k=1, kernel=5))
    assert st == F.OK
    assert rel_err(got, ref) < TOL[prec]


@pytest.mark.parametrize("exponent", [2, -130, 90])
def test_mixed_differences_outside_float_range(exponent):
    """A linear problem scales: u0 2^e gives u 2^e.  At 2^-130 every difference is subnormal in float (the
    conversions take the hardware path; quantum 2^-149, so relative 2^-19 of the largest value a stage and
    at most s Q of that over a step: below 1e-3 for s = 4); at 2^2 and 2^90 the bits scale exactly."""
    shape, s = (7, 9, 35), 4
    u0, field = seeded_case(shape, "dirichlet", "field", 77)
    u0[:, :4] = 0.0  # equal neighbours too
    opr = oracle_problem(3, "dirichlet", "field", 1.0, field.astype(np.float32).astype(np.float64))
    dt = 0.9 * O.beta(s) / O.rho_bound(opr, u0)
    kt = torch.as_tensor(field, dtype=torch.float32, device="cuda")
    pr = F.make_problem(3, tuple(reversed(shape)), 1.0, "dirichlet", "field", "mixed", kappa_field=kt)
    plan = F.frkc2_plan(s)
    base, st0 = run(pr, plan, u0, dt, 1, "mixed")
    got, st = run(pr, plan, np.ldexp(u0, exponent), dt, 1, "mixed")
    assert st0 == F.OK and st == F.OK
    got = np.ldexp(got, -exponent)
    if exponent > 0:
        assert np.array_equal(got, base)
    else:
        assert rel_err(got, base) < 1e-3


def test_mixed_nonfinite_is_reported():
    u0, field = seeded_case((5, 8, 40), "periodic", "field", 78)
    u0[2, 3, 7] = np.inf
    kt = torch.as_tensor(field, dtype=torch.float32, device="cuda")
    pr = F.make_problem(3, (40, 8, 5), 1.0, "periodic", "field", "mixed", kappa_field=kt)
    got, st = run(pr, F.frkc2_plan(4), u0, 1e-3, 1, "mixed")
    assert st == F.ENONFINITE and not np.isfinite(got).all()
