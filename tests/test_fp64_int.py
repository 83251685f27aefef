"""The FP64 functions on the integer pipe (fp64_int.cuh) against long double, on the host and
on the device, whose FP32 seeds differ from the host's.

Bounds, from the arithmetic of each (ulp: a unit in the last place of the exact result; seeds to
2^-21 relative, so e <= 2^-20): inverse root and reciprocal end at e^3 and a few units of
2^-62, below 2^-59 relative or 1/64 ulp before the one rounding; the exponential carries 2^-62;
a product loses one unit of 2^-63. The logarithm sums e ln2 and ln m at 2^-55 (at 2^-62 for
1/2 <= x < 2): (1 + |e|/2) 2^-55 beside a result of at least 0.69 |e|, or 0.54 ulp, and the
rounding; near 1 the bound is absolute. The Hernquist factor multiplies four such
values (1/16 ulp). The NFW mass factor is a difference of terms at 2^-62, of which u = 1 - t
brings 2^-60: 12 2^-62 absolute between t = q/(1+q) = 2^-7 and q = 1, 2 ulp beyond (2^-56 beside
0.19 and more), and 2 ulp of its FP64 series below."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FN = dict(sqrt=0, rsqrt=1, div=2, mul=3, exp=4, exp_mhalf=5, log=6, hernquist=7, nfw_mu=8)
DEVICE = [pytest.param(0, id="host"), pytest.param(1, id="device", marks=pytest.mark.gpu)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1202_2355_gb300 import build
    so = str(tmp_path_factory.mktemp("int") / "libint.so")
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", build.ARCH, "-ftz=true", "-prec-div=false", "-prec-sqrt=false",
                    "-fmad=false", "-Xcompiler", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_1202_2355_gb300", "csrc"), "-o", so,
                    os.path.join(ROOT, "tests", "kernels", "int_check.cu")], check=True)
    L = C.CDLL(so)
    L.int_check.argtypes = [C.c_int, C.c_int, C.c_void_p, C.c_longlong, C.c_void_p, C.c_void_p]
    L.int_seed_bits.argtypes, L.int_seed_bits.restype = [C.c_float], C.c_ulonglong
    L.int_leads.argtypes = [C.c_void_p]
    return L


def _run(lib, fn, device, a, b=1.0, c=1.0, errors=True):
    a, b, c = np.broadcast_arrays(np.asarray(a, np.float64), np.asarray(b, np.float64), np.asarray(c, np.float64))
    x = np.ascontiguousarray(np.concatenate([a, b, c]))
    y, err = np.empty(a.size), np.empty(a.size)
    assert lib.int_check(FN[fn], device, x.ctypes.data, a.size, y.ctypes.data, err.ctypes.data if errors else None) == 0
    return y, err


def _significands(rng, n):
    """Significands in [1, 2), with those next to 1, to 2 and to round numbers among them."""
    m = 1.0 + rng.random(n)
    k = np.arange(1, 200)
    edge = np.concatenate([1.0 + k * 2.0 ** -52, 2.0 - k * 2.0 ** -52, 1.0 + k / 256.0, 1.0 + k / 256.0 - 2.0 ** -52])
    edge = np.concatenate([edge, 1.0 + k * 2.0 ** -23, 2.0 - k * 2.0 ** -23, 2.0 - k * 2.0 ** -23 + 2.0 ** -50])
    return np.concatenate([m, edge[(edge >= 1) & (edge < 2)], [1.0]])


def _positive(rng, n, lo=-199, hi=200):
    m = _significands(rng, n)
    return np.ldexp(m, rng.integers(lo, hi, m.size))


def test_seeds_stay_in_their_range(lib):
    """A seed just below 1/2 or above 1 - 2^-24 gives the nearest end, not a misread significand."""
    lo, hi, f = 0x800000, 0xffffff, np.float32
    for y in (f(0.5), np.nextafter(f(0.5), f(0)), f(0.5) * (f(1) - f(2.0 ** -21)), f(0.4999)):
        assert lib.int_seed_bits(y) == lo, y
    for y in (np.nextafter(f(1), f(0)), f(1), np.nextafter(f(1), f(2)), f(1.0001)):
        assert lib.int_seed_bits(y) == hi, y
    assert lib.int_seed_bits(f(0.75)) == 0xc00000


@pytest.mark.gpu
def test_every_lead_on_the_device(lib):
    """Reciprocal and inverse root from every FP32 seed the device can give: within 2^-59 (the
    inverse root's residual is twice its error)."""
    out = (C.c_ulonglong * 2)()
    assert lib.int_leads(out) == 0
    assert out[0] <= 2 and out[1] <= 4, list(out)


@pytest.mark.parametrize("device", DEVICE)
@pytest.mark.parametrize("fn,bound", [("sqrt", 0.5 + 2 ** -5), ("rsqrt", 0.5 + 2 ** -5)])
def test_roots(lib, fn, bound, device):
    x = _positive(np.random.default_rng(1), 400_000)
    y, err = _run(lib, fn, device, x)
    assert err.max() <= bound, (err.max(), x[err.argmax()])


@pytest.mark.parametrize("device", DEVICE)
@pytest.mark.parametrize("fn,bound", [("div", 0.5 + 2 ** -5), ("mul", 0.501)])
def test_products_and_quotients(lib, fn, bound, device):
    rng = np.random.default_rng(2)
    a, b = _positive(rng, 400_000), _positive(rng, 400_000)
    a = a * rng.choice([-1.0, 1.0], a.size)
    b = rng.permutation(b) if fn == "div" else rng.permutation(b) * rng.choice([-1.0, 1.0], b.size)
    y, err = _run(lib, fn, device, a, b)
    assert err.max() <= bound, (err.max(), a[err.argmax()], b[err.argmax()])


@pytest.mark.parametrize("device", DEVICE)
def test_exponentials(lib, device):
    rng = np.random.default_rng(3)
    L = np.log(2.0) / 256
    x = np.concatenate([rng.uniform(-707, 709, 300_000), rng.uniform(-1, 1, 100_000), rng.normal(size=50_000) * 1e-6,
                        (np.arange(-4000, 4000) + 0.5) * L, np.arange(-4000, 4000) * L, [0.0, -0.0, 708.99, -706.99]])
    y, err = _run(lib, "exp", device, x)
    assert err.max() <= 0.5 + 2 ** -5, (err.max(), x[err.argmax()])
    t = np.concatenate([rng.uniform(0, 1400, 200_000), np.exp(rng.uniform(-40, 3, 200_000)), [0.0, -0.0, 5e-324, 1e-300]])
    y, err = _run(lib, "exp_mhalf", device, t)
    assert err.max() <= 0.5 + 2 ** -5, (err.max(), t[err.argmax()])


@pytest.mark.parametrize("device", DEVICE)
def test_logarithm(lib, device):
    x = _positive(np.random.default_rng(4), 400_000)
    y, err = _run(lib, "log", device, x)
    far = (x < 0.5) | (x >= 2.0)
    assert err[far].max() <= 1.1, (err[far].max(), x[far][err[far].argmax()])
    x = np.ldexp(_significands(np.random.default_rng(5), 400_000), np.random.default_rng(6).integers(-1, 1, 1))
    x = np.concatenate([x, x / 2, 1 + np.linspace(-1e-6, 1e-6, 20001)])
    x = x[(x >= 0.5) & (x < 2.0)]
    y, err = _run(lib, "log", device, x)
    r = np.abs(np.log(x))
    ulp = np.where(r > 0, np.spacing(r), 0.0)
    assert np.all(err * ulp <= 2.0 ** -60 + 0.5 * ulp)


@pytest.mark.parametrize("device", DEVICE)
def test_force_factors(lib, device):
    rng = np.random.default_rng(7)
    r2 = np.concatenate([np.exp(rng.uniform(-30, 30, 300_000)), _positive(rng, 20_000, -100, 100)])
    gm, a = np.exp(rng.uniform(-5, 5, r2.size)), np.exp(rng.uniform(-5, 5, r2.size))
    y, err = _run(lib, "hernquist", device, r2, gm, a)
    assert err.max() <= 0.5 + 2 ** -4, (err.max(), r2[err.argmax()])
    rs = np.exp(rng.uniform(-3, 3, 400_000))
    q = np.concatenate([np.exp(rng.uniform(-25, 25, 300_000)), 2.0 ** -7 / (1 - 2.0 ** -7) * (1 + rng.normal(size=100_000) * 0.05)])
    y, err = _run(lib, "nfw_mu", device, q * rs, rs)
    t = q * rs / (rs + q * rs)
    ulp = np.spacing(y)
    mid = (t >= 2.0 ** -7 * (1 - 1e-12)) & (q <= 1.0)
    assert np.all(err[mid] * ulp[mid] <= 12 * 2.0 ** -62 + ulp[mid]), (err[mid] * ulp[mid]).max() * 2.0 ** 62
    assert err[~mid].max() <= 2.0, (err[~mid].max(), q[~mid][err[~mid].argmax()])


@pytest.mark.parametrize("device", DEVICE)
def test_special_values(lib, device):
    """Out of the functions' ranges: the results of the FP64 operations."""
    inf, nan, sub = np.inf, np.nan, 5e-324
    odd = np.array([0.0, -0.0, sub, 1e-310, 1e-308, 1e300, 1.7e308, inf, -inf, nan, -nan, 1.0, -1.0, 3.7])
    with np.errstate(all="ignore"):
        a, b = (v.ravel() for v in np.meshgrid(odd, odd))
        want = a * b
        y, _ = _run(lib, "mul", device, a, b, errors=False)
        big = np.isfinite(want) & (np.abs(want) > 0)
        assert np.array_equal(np.isnan(y), np.isnan(want)) and np.array_equal(y[~big & ~np.isnan(y)], want[~big & ~np.isnan(y)])
        assert np.all(np.abs(y[big] - want[big]) <= np.spacing(np.abs(want[big])))
        b = np.abs(b)  # the divisor is positive
        want = a / b
        y, _ = _run(lib, "div", device, a, b, errors=False)
        big = np.isfinite(want) & (np.abs(want) > 0)
        assert np.array_equal(np.isnan(y), np.isnan(want)) and np.array_equal(y[~big & ~np.isnan(y)], want[~big & ~np.isnan(y)])
        assert np.all(np.abs(y[big] - want[big]) <= np.spacing(np.abs(want[big])))
        y, _ = _run(lib, "sqrt", device, odd, errors=False)
        assert np.allclose(y, np.sqrt(odd), rtol=2e-16, atol=0, equal_nan=True)
        y, _ = _run(lib, "log", device, odd, errors=False)
        assert np.allclose(y, np.log(odd), rtol=1e-15, atol=0, equal_nan=True)
    y, _ = _run(lib, "exp", device, [-inf, -1e300, -745.2, -708.0, -707.0, inf, 710.0, 1e300, nan], errors=False)
    assert np.all(y[:5] == 0.0) and np.all(np.isposinf(y[5:8])) and np.isnan(y[8])
    y, _ = _run(lib, "exp_mhalf", device, [inf, 1414.0, 1e300, 0.0, -0.0, sub], errors=False)
    assert np.all(y[:3] == 0.0) and np.all(y[3:] == 1.0)
    # NaN of either sign (an invalid operation gives the negative one on the device) stays NaN
    y, _ = _run(lib, "exp_mhalf", device, np.array([0x7ff8 << 48, 0xfff8 << 48, (0xfff << 52) | 1], np.uint64).view(np.float64),
                errors=False)
    assert np.all(np.isnan(y)), y
