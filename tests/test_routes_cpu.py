"""Which kernels a call launches, and with which grids, without a GPU: the library's host code over a stand-in runtime
that checks launches against the limits of the real one (fake_runtime.py)."""
import ctypes
import math
import random
import time

import pytest

import fake_runtime as R


@pytest.fixture(scope="module")
def F(tmp_path_factory):
    return R.load(str(tmp_path_factory.mktemp("fake")))


def bruss(F, nx, ny, prec, s=16, nsteps=1, bc="periodic", tune=None):
    p = F.make_bruss_problem((nx, ny), bc=bc, precision=prec)
    ws = R.Buffer(F.frkc2_bruss_workspace_size(p), 1 << 41)
    F._lib.fake_reset()
    F.frkc2_bruss_step(F.frkc2_plan(s), p, 1e-4, nsteps, 0.0, R.Buffer(1), R.Buffer(1, 1 << 42), ws, tune, stream=0)
    return R.launches(F)


@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("nx,ny", [(16, 2_000_000), (1, 1 << 24), (256, 4_000_000), (4_000_000, 256), (16, 1_400_000), (200, 200)])
def test_bruss_fp32_takes_tall_grids(F, nx, ny, bc):
    """Passes with a CTA for each of their regions, or the persistent kernel where these have too many rows."""
    got = bruss(F, nx, ny, "fp32", bc=bc)
    assert {g.kernel for g in got} == ({"k_bruss2d"} if ny >= 2_000_000 else {"k_bruss_tb2d"})
    for g in got:
        edge = 16 * (2 if "ILi2E" in g.mangled else 4)
        assert g.cooperative or any(g.grid[:2] == (-(-nx // (edge - 2 * k)), -(-ny // (edge - 2 * k))) for k in range(1, 9))


def step(F, n, prec, bc="periodic", kappa="const", s=16, nsteps=1, tune=None):
    p = F.make_problem(len(n), n, 1.0, bc, kappa, prec)
    if kappa == "field":
        p.kappa = 1 << 43
    ws = R.Buffer(F.frkc2_workspace_size(p), 1 << 41)
    F._lib.fake_reset()
    F.frkc2_step(F.frkc2_plan(s), p, 1e-4, nsteps, 0.0, R.Buffer(1), ws, tune, stream=0)
    return R.launches(F)


@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
@pytest.mark.parametrize("nx,ny", [(12, 2_000_000), (16, 1_500_000), (24, 1_400_000), (1, 3_000_000), (301, 3_900_000), (100, 100)])
def test_fp32_2d_takes_tall_grids(F, nx, ny, bc):
    """Every pass has a CTA for each of its regions, however many rows of them there are."""
    got = [g for g in step(F, (nx, ny), "fp32", bc, s=32) if g.kernel != "k_faces_padded"]
    assert {g.kernel for g in got} == {"k_tb2d_reg"}
    edge = 16 * (2 if "ILi2E" in got[0].mangled else 4)
    for g in got:
        assert any(math.prod(g.grid) == -(-nx // (edge - 2 * k)) * -(-ny // (edge - 2 * k)) for k in range(1, 13))


def adjoint(F, n, prec, s, nsteps, ckpt, bc="periodic"):
    p = F.make_problem(len(n), n, 1.0, bc, "field", prec)
    p.kappa = 1 << 50
    plan = F.frkc2_plan(s)
    ws = R.Buffer(F.frkc2_adjoint_workspace_size(plan, p, nsteps, ckpt), 1 << 41)
    F._lib.fake_reset()
    F.frkc2_adjoint(plan, p, 1e-4, nsteps, ckpt, *(R.Buffer(1, (42 + i) << 40) for i in range(4)), ws, stream=0)
    return R.launches(F)


@pytest.mark.parametrize("nx,ny", [(8, 2_900_000), (2, 3_000_000), (100, 3_100_000), (100, 100)])
def test_fp32_adjoint_takes_tall_grids(F, nx, ny):
    got = adjoint(F, (nx, ny), "fp32", 20, 2, 1)
    tb = [g for g in got if g.kernel in ("k_tape_tb2d", "k_adjrev_tb2d")]
    assert {g.kernel for g in tb} == {"k_tape_tb2d", "k_adjrev_tb2d"}
    for g in tb:
        assert any(math.prod(g.grid) == -(-nx // (64 - 2 * k)) * -(-ny // (64 - 2 * k)) for k in range(1, 13))


def test_second_device(F):
    """Calls on a second GPU of the process launch what they launch on the first (a kernel's shared memory limit is set on
    each device)."""
    def runs():
        out = []
        for prec in ("fp64", "fp32", "mixed", "dfloat"):
            for n in ((100, 90), (700, 611)):
                out.append(lambda n=n, prec=prec: step(F, n, prec, kappa="field"))
                out.append(lambda n=n, prec=prec: step(F, n, prec, "dirichlet", tune=F.make_tuning(k=1)))
        for prec in ("fp64", "fp32"):
            out += [lambda prec=prec: bruss(F, 120, 90, prec), lambda prec=prec: adjoint(F, (120, 90), prec, 16, 2, 1)]
        p = F.make_problem(2, (90, 80), 1.0, "periodic", "const", "fp64")
        ws, plan = R.Buffer(F.frkc2_workspace_size(p), 1 << 41), F.frkc2_plan(16, flags=F.PLAN_PAIRED)
        out.append(lambda: (F._lib.fake_reset(), F.frkc2_step(plan, p, 1e-4, 1, 0.0, R.Buffer(1), ws, stream=0), R.launches(F))[2])
        return out

    for run in runs():
        first = run()
        try:
            F._lib.cudaSetDevice(1)
            second = run()
        finally:
            F._lib.cudaSetDevice(0)
        assert [g._replace(device=1) for g in first] == second and {g.device for g in second} == {1}


@pytest.mark.parametrize("error", [720, 801, 701])  # too large for a cooperative launch, not supported, out of resources
def test_refused_cooperative_launch(F, error):
    """Where the context refuses the whole job in one launch, a call takes the launch per stage (the Brusselator, whose
    other form is cooperative too, still says so)."""
    def kernels(run):
        return {g.kernel for g in run()}

    calls = [lambda: step(F, (100, 90), "fp64", kappa="field"), lambda: adjoint(F, (100, 90), "fp64", 16, 4, 1)]
    plain = [kernels(c) for c in calls]
    assert all("k_resident2d" in k for k in plain)
    F._lib.fake_refuse_cooperative(error)
    try:
        assert kernels(calls[0]) == {"k_faces", "k_face_pairs", "k_stream2d"}
        assert kernels(calls[1]) == plain[1] - {"k_resident2d"}
        with pytest.raises(F.Frkc2Error):
            bruss(F, 100, 90, "fp64")
        assert len(bruss(F, 100, 90, "fp64", tune=F.make_tuning(kernel=2))) == 16
    finally:
        F._lib.fake_refuse_cooperative(0)
    assert [kernels(c) for c in calls] == plain


@pytest.mark.parametrize("prec,n,kernel", [("fp32", (2048, 300_000, 1), "k_stream3d"), ("fp32", (2048, 200_000, 2), "k_stream3d_f32"),
                                           ("fp32", (70_000, 70_000, 1), "k_stream3d"), ("fp64", (70_000, 70_000, 1), "k_stream3d"),
                                           ("mixed", (16_000, 300_000, 1), "k_stream3d")])
def test_3d_streams_planes_of_any_size(F, prec, n, kernel):
    got = step(F, n, prec, kappa="power", s=4)
    assert [g.kernel for g in got] == [kernel] * 4


def chunks(F):
    f = F._lib._ZN5frkc215stream3d_chunksExix
    f.argtypes, f.restype = [ctypes.c_longlong, ctypes.c_int, ctypes.c_longlong], ctypes.c_int
    return f


def test_3d_chunks_are_the_best_of_all_counts(F):
    """The number of chunks along z is that of a look at every count: fewest planes over its waves, then fewest chunks."""
    f, r = chunks(F), random.Random(3)
    for _ in range(3000):
        nz, slots = int(math.exp(r.uniform(0, 7))), 152 * r.randint(1, 8)
        blocks = int(math.exp(r.uniform(0, 9)))
        planes = [(-(-blocks * c // slots) * (-(-nz // c) + 2), c) for c in range(1, min(nz, 256) + 1)]
        assert f(blocks, nz, slots) == min(planes)[1], (blocks, nz, slots)


def test_3d_chunks_cost_a_launch_little(F):
    """Every stage asks: a tall box takes about the time of a flat one, most of it the call from here."""
    f = chunks(F)

    def us(nz):
        best = math.inf
        for _ in range(30):
            t = time.perf_counter()
            for _ in range(500):
                f(3, nz, 608)
            best = min(best, (time.perf_counter() - t) / 500 * 1e6)
        return best

    assert us(250) < 2 * us(1)


# The sizes at which the GPU tests compare these kernels with others, and some on the other side of each rule.
@pytest.mark.parametrize("s", [6, 16, 1024])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 9), (9, 1), (16, 4), (15, 16), (33, 21), (64, 64), (7, 300), (300, 7), (200, 200), (256, 256),
                                   (400, 400), (34, 411), (457, 355), (247, 777), (619, 305)])
def test_bruss_fp64_small_grids_in_registers(F, nx, ny, s):
    got = bruss(F, nx, ny, "fp64", s=s, nsteps=2)
    assert [(g.kernel, g.cooperative) for g in got] == [("k_bruss_resident", True)]
    assert got[0].grid[0] <= 152


@pytest.mark.parametrize("nx,ny,s", [(500, 512, 16), (610, 600, 16), (420, 269, 16), (2048, 2048, 16), (64, 64, 1026)])
def test_bruss_fp64_larger_grids_persistent(F, nx, ny, s):
    assert {g.kernel for g in bruss(F, nx, ny, "fp64", s=s)} == {"k_bruss2d"}


@pytest.mark.parametrize("nx,ny,s,passes", [(2, 3, 4, 2), (24, 20, 16, 2), (96, 33, 10, 2), (144, 144, 16, 2), (700, 611, 12, 3),
                                            (2048, 1030, 16, 2)])
def test_bruss_fp32_stages_in_few_passes(F, nx, ny, s, passes):
    assert [g.kernel for g in bruss(F, nx, ny, "fp32", s=s)] == ["k_bruss_tb2d"] * passes


@pytest.mark.parametrize("nx,ny,s,nsteps,ckpt,plain", [(5, 8, 6, 4, 1, 3), (33, 21, 16, 5, 2, 2), (97, 130, 32, 4, 1, 3), (200, 200, 16, 7, 3, 2),
                                                       (700, 700, 16, 2, 1, 0), (33, 21, 16, 5, 5, 0)])
def test_fp64_adjoint_forward_segments_in_one_launch(F, nx, ny, s, nsteps, ckpt, plain):
    """Every segment but the last runs forward in one launch where the grid fits."""
    assert [g.kernel for g in adjoint(F, (nx, ny), "fp64", s, nsteps, ckpt)].count("k_resident2d") == plain
