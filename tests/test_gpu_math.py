"""The square roots, kappa(w) = 1 + c w^2.5 and the conversions of frkc2_math.cuh on their own, against correctly rounded or
extended results: the whole normal range of the roots, all quadrants and axes of w, moduli whose square is below the smallest
normal number and zero, and the bits of the conversions."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1702_03818_gb300 import build as B

    out = str(tmp_path_factory.mktemp("math") / "libmath.so")
    subprocess.run([B._nvcc(), *B.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", B.CSRC, "-I", B.INCLUDE,
                    os.path.join(HERE, "math_kernels.cu"), "-o", out], check=True)
    return C.CDLL(out)


def call(f, inputs, scalars, outputs):
    """f(inputs on the GPU, scalars, outputs, count) -> the outputs as arrays."""
    n = len(inputs[0])
    dev = [torch.as_tensor(a, device="cuda") for a in inputs]
    out = [torch.empty(n, dtype=t, device="cuda") for t in outputs]
    torch.cuda.synchronize()
    assert f(*(C.c_void_p(t.data_ptr()) for t in dev), *scalars, *(C.c_void_p(t.data_ptr()) for t in out), C.c_int(n)) == 0
    return [t.cpu().numpy() for t in out]


def test_roots(lib):
    """e = 1 - a y^2 of the seed is below 2^-18 (its 20 bits), so the series' next term, 5 e^3 / 16, is below 2^-55; the rounding
    of t = a y reaches the result by half, and the last operation rounds: 2^-54 + 2^-53 + 2^-55, below 2^-52."""
    r = np.random.default_rng(1)
    a = np.ldexp(r.uniform(1.0, 2.0, 1 << 18), r.integers(-1022, 1024, 1 << 18))
    a = np.concatenate([a, np.ldexp(1.0 + np.arange(4096) / 4096.0, 1), np.ldexp(1.0 + np.arange(4096) / 4096.0, -2), [2.0 ** -1022, np.finfo(float).max]])
    s, q = call(lib.run_roots, [a], [], [torch.float64, torch.float64])
    root = np.sqrt(a.astype(np.longdouble))
    assert np.max(np.abs(s / root - 1)) < 2.0 ** -52
    assert np.max(np.abs(q * root - 1)) < 2.0 ** -52


def points(dtype, most, n=1 << 16):
    """States w = x + i y: moduli over the range in which |w|^2 and w^2.5 are normal, in every direction, on the axes with both zeros,
    and small and zero ones."""
    r = np.random.default_rng(2)
    th, m = r.uniform(-np.pi, np.pi, n), np.ldexp(r.uniform(1, 2, n), r.integers(-most, most, n))
    x, y = m * np.cos(th), m * np.sin(th)
    near = r.uniform(0.5, 2.0, n)  # the states of a run: about 1, small imaginary parts
    x, y = np.concatenate([x, near, -near]), np.concatenate([y, near * r.uniform(-1e-3, 1e-3, n), near * r.uniform(-1e-3, 1e-3, n)])
    ax = np.array([0.0, -0.0, 1.0, -1.0, 2.0, -2.0, 0.3, -0.3])
    tiny = np.array([0.0, 1.0, -1.0]) * float(np.finfo(dtype).tiny)
    gx, gy = (g.ravel() for g in np.meshgrid(np.concatenate([ax, tiny, tiny / 8]), np.concatenate([ax, tiny, tiny / 8])))
    x, y = np.concatenate([x, gx, gx]), np.concatenate([y, gy, gy])
    return x.astype(dtype)[: len(x) // 2 * 2], y.astype(dtype)[: len(y) // 2 * 2]


def kappa(x, y, c):
    """1 + c w^2.5 in extended precision (the sign of a zero imaginary part selects the side of the cut)."""
    x, y = x.astype(np.longdouble), y.astype(np.longdouble)
    m = np.hypot(x, y)
    t = np.sqrt((m + np.abs(x)) / 2)
    h = np.divide(np.abs(y), 2 * t, out=np.zeros_like(t), where=t > 0)
    sr, si = np.where(x >= 0, t, h), np.copysign(np.where(x >= 0, h, t), y)
    qr, qi = (x - y) * (x + y), 2 * x * y
    return 1 + c * (qr * sr - qi * si), c * (qr * si + qi * sr), abs(c) * m ** 2.5


def check(got, x, y, c, u, bound):
    kr, ki, size = kappa(x, y, c)
    off = np.maximum(np.abs(got[0] - kr), np.abs(got[1] - ki)) / (1 + size)
    worst = int(np.argmax(off))
    assert off[worst] < bound * u, (x[worst], y[worst], float(off[worst] / u))


@pytest.mark.parametrize("c", [1.0, 0.37, -0.2])
def test_kappa_fp64(lib, c):
    """Roundings of u = 2^-53 each: |w|^2 2, r 2.5, r + |x| 3.5, its reciprocal root 3.3, the square root's parts 8, w^2 2, their
    products 11 in two terms of at most |w|^2.5 each, c 2: below 32 u of 1 + |c| |w|^2.5."""
    x, y = points(np.float64, 400)
    check(call(lib.run_kappa64, [x, y], [C.c_double(c)], [torch.float64] * 2), x, y, c, 2.0 ** -53, 32)


@pytest.mark.parametrize("c", [1.0, 0.37, -0.2])
@pytest.mark.parametrize("form", ["pair", "mixed"])
def test_kappa_fp32(lib, form, c):
    """As in FP64 with u = 2^-24 and the reciprocal root within 2^-22.9, 2.2 u, of exact where that was 1.5: below 32 u."""
    x, y = points(np.float32, 45)
    c = float(np.float32(c))
    f = lib.run_kappa32 if form == "pair" else lib.run_kappa_mixed
    check(call(f, [x, y], [C.c_float(c)], [torch.float32] * 2), x, y, c, 2.0 ** -24, 32)


def test_kappa_nan_and_infinity_do_not_vanish(lib):
    bad = np.array([np.nan, -np.nan, np.inf, -np.inf, 1.0, 0.0])
    x, y = (g.ravel() for g in np.meshgrid(bad, bad))
    at = ~(np.isfinite(x) & np.isfinite(y))
    for f, dtype, ct, t in ((lib.run_kappa64, np.float64, C.c_double, torch.float64), (lib.run_kappa32, np.float32, C.c_float, torch.float32),
                            (lib.run_kappa_mixed, np.float32, C.c_float, torch.float32)):
        kr, ki = call(f, [x.astype(dtype), y.astype(dtype)], [ct(1.0)], [t] * 2)
        assert not (np.isfinite(kr[at]) & np.isfinite(ki[at])).any()


def test_conversions_are_the_hardwares_bits(lib):
    """Every bit pattern: where the value or its float is not normal (zero apart) the call asks for the hardware's conversion."""
    r = np.random.default_rng(3)
    n = 1 << 20
    d = r.integers(0, 1 << 64, n, dtype=np.uint64, endpoint=False).view(np.float64).copy()
    e = np.ldexp(r.uniform(1, 2, n // 2), r.integers(-160, 140, n // 2)) * r.choice([-1.0, 1.0], n // 2)  # in and around float's range
    ties = np.float32(r.uniform(1, 2, n // 4)).astype(np.float64) + 2.0 ** -24  # halfway between two floats
    d[: n // 2], d[n // 2: n // 2 + n // 4] = e, ties
    d[-8:] = [0.0, -0.0, np.inf, -np.inf, np.nan, 2.0 ** -126, 2.0 ** -126 * (1 - 2.0 ** -30), float(np.finfo(np.float32).max) * (1 + 2.0 ** -26)]
    f = r.integers(0, 1 << 32, n, dtype=np.uint32, endpoint=False).view(np.float32).copy()
    f[:6] = [0.0, -0.0, np.inf, np.nan, 2.0 ** -126, 2.0 ** -149]
    nd, wf, slow = call(lib.run_convert, [d, f], [], [torch.float32, torch.float64, torch.uint8])
    with np.errstate(over="ignore", invalid="ignore"):
        want = d.astype(np.float32)
    tiny = 2.0 ** -126
    asks = ~((d == 0) | ((np.abs(d) >= tiny) & (np.abs(d) < 2.0 ** 128)))
    assert np.array_equal(slow & 1 == 1, asks)
    assert np.array_equal(nd[~asks].view(np.uint32), want[~asks].view(np.uint32))
    asks = ~((f == 0) | ((np.abs(f) >= np.float32(tiny)) & np.isfinite(f)))
    assert np.array_equal(slow & 2 == 2, asks)
    assert np.array_equal(wf[~asks].view(np.uint64), f[~asks].astype(np.float64).view(np.uint64))
