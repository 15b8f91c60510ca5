"""The device arithmetic that stands in for divisions, roots and conversions in
FP64 (dfv_device.cuh), function by function over its range: at the points
where a series gives way to a closed form, at ties, zeros, subnormals,
infinities and NaN.  Conversions and comparisons have one right answer; the
bounds of the others are counted from their roundings (u = 2^-53):
  m_rcp        one rounding, and the iteration's remainder far below it: 1 u,
               allowed 2 u (one unit in the last place)
  m_div        m_rcp and a product: 2 u, allowed 3 u; m_quot likewise
  m_sqrt       half the product's rounding and the last one: 1.5 u, allowed 2 u
  m_sqrt_ratio two roundings halved, two whole: 3 u, allowed 4 u
  m_whole_pow  x^8: 7 u, allowed 8 u
  series       each Horner step rounds a term far below the sum's: 2 u, allowed 3 u
  closed forms of y: cosh and sinh by e^y and 1/e^y, (1 ulp each and a difference
               that loses a factor of at most 1/tanh y): (4 + 4/y) u; artanh(z)/z by
               the logarithm of (1 + z)/(1 - z), whose relative error is an absolute
               one of the logarithm, 2 artanh z: (4 + (4 + 2 z/(1 - z))/(2 artanh z)) u"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
HERE = os.path.dirname(os.path.abspath(__file__))
NAMES = ["rcp", "div", "quot", "sqrt", "sqrt_ratio", "artanh", "cosh", "sinhc", "expm1", "widen", "narrow", "min",
         "max", "pred", "less", "power"]
INF, NAN = np.inf, np.nan
TINY, HUGE = np.finfo(float).tiny, np.finfo(float).max
EDGES = np.array([0.0, 5e-324, 1e-310, TINY, 1e-300, 1e-290, 1e-160, 1.0 - U, 1.0, 1.0 + 2 * U, 3.0, 1e160, 1e300,
                  HUGE, INF])


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2111_11806_gb300 import _build
    so = str(tmp_path_factory.mktemp("device_math") / "libdevice_math.so")
    subprocess.check_call([_build.nvcc()] + _build.ARCH + _build.FLAGS
                          + ["-I" + _build.CSRC, "-shared", "-o", so, os.path.join(HERE, "device_math.cu"), "-lcudart"])
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def dev(lib):
    dp = ctypes.POINTER(ctypes.c_double)

    def call(name, a, b=None):
        a = np.ascontiguousarray(a, dtype=np.float64)
        b = np.ascontiguousarray(np.ones_like(a) if b is None else b, dtype=np.float64)
        out = np.empty_like(a)
        st = lib.dm_eval(NAMES.index(name), a.ctypes.data_as(dp), b.ctypes.data_as(dp), out.ctypes.data_as(dp), a.size)
        assert st == 0, st
        return out
    return call


def spread(seed, lo, hi, n=200000):
    """Numbers of both signs, spread over their exponents from 2^lo to 2^hi."""
    rng = np.random.default_rng(seed)
    return rng.choice((-1.0, 1.0), n) * np.exp2(rng.uniform(lo, hi, n))


def close(got, want, bound):
    """|got - want| <= bound |want| in extended precision."""
    d = np.abs(got.astype(np.longdouble) - want)
    assert np.all(d <= np.longdouble(1.0) * bound * np.abs(want)), float(np.max(d / np.abs(want)) / U)


def same(got, want):
    """Equal bits, all NaNs alike."""
    ok = (got.view(np.uint64) == want.view(np.uint64)) | (np.isnan(got) & np.isnan(want))
    assert np.all(ok), (got[~ok][:4], want[~ok][:4])


def test_reciprocal_and_quotients(dev):
    x = spread(1, -1021, 1021)
    close(dev("rcp", x), 1 / x.astype(np.longdouble), 2 * U)
    a, b = spread(2, -500, 500), spread(3, -500, 500)
    close(dev("div", a, b), a.astype(np.longdouble) / b, 3 * U)
    close(dev("quot", a, b), a.astype(np.longdouble) / b, 3 * U)
    with np.errstate(all="ignore"):
        # zeros, infinities and the subnormals whose reciprocal overflows, as a division gives them
        e = np.array([0.0, -0.0, INF, -INF, NAN, 5e-324, -1e-310])
        same(dev("rcp", e), 1 / e)
        # quotients of subnormals, correctly rounded
        s = spread(4, -1074, -1019)
        same(dev("quot", s, s[::-1].copy()), s / s[::-1])
        same(dev("quot", np.zeros(3), np.array([5e-324, -1e-310, TINY])), np.array([0.0, -0.0, 0.0]))


def test_square_roots(dev):
    x = np.abs(spread(5, -1074, 1023))
    close(dev("sqrt", x), np.sqrt(x.astype(np.longdouble)), 2 * U)
    with np.errstate(all="ignore"):
        e = np.concatenate([EDGES, [1e-290 * (1 - U), -1.0, -INF, NAN]])
        got, want = dev("sqrt", e), np.sqrt(e)
        assert np.all((np.abs(got - want) <= 2 * U * want) | (got == want) | (np.isnan(got) & np.isnan(want))), got
    # a ratio in range of products that leave it: up to 2^-1600 and 2^1600
    for lo, hi in ((-300, 300), (-800, -500), (500, 800)):
        a, b = np.abs(spread(6, lo, hi)), np.abs(spread(7, lo, hi))
        close(dev("sqrt_ratio", a, b), np.sqrt(a.astype(np.longdouble) / b), 4 * U)
    b = np.array([1.0, 1e-200, 1e200])
    same(dev("sqrt_ratio", np.zeros(3), b), np.zeros(3))
    assert np.all(np.isnan(dev("sqrt_ratio", np.array([-1.0, -1e-200, NAN]), b)))


def test_series_and_closed_forms(dev):
    L = np.longdouble
    near = np.array([1 - 2 * U, 1.0, 1 + 4 * U])
    z2 = np.concatenate([np.linspace(0, 0.0101, 20001)[1:], 0.01 * near, np.linspace(0.01, 0.9, 20001),
                         [1e-300, 1e-30]])
    z = np.sqrt(z2.astype(L))
    want = 0.5 * (np.log1p(z) - np.log1p(-z)) / z
    close(dev("artanh", z2), want, np.where(z2 < 0.01, 3.0, 4 + (4 + 2 * z / (1 - z)) / (2 * z * want)) * U)
    y2 = np.concatenate([np.linspace(0, 0.0201, 20001)[1:], 0.02 * near, np.linspace(0.02, 9.0, 20001),
                         [1e-300, 1e-30]])
    y = np.sqrt(y2.astype(L))
    # sinh(y)/y without the difference for small y
    sinhc = np.where(y < 0.5, 1 + y * y / 6 * (1 + y * y / 20 * (1 + y * y / 42 * (1 + y * y / 72 * (1 + y * y / 110 * (
        1 + y * y / 156 * (1 + y * y / 210 * (1 + y * y / 272))))))), np.sinh(y) / y)
    bound = np.where(y2 < 0.02, 3.0, 4 + 4 / y) * U
    close(dev("cosh", y2), np.cosh(y), bound)
    close(dev("sinhc", y2), sinhc, bound)
    x = np.concatenate([np.linspace(-0.0625, 0.0625, 20001), [1e-300, 1e-30, -1e-17]])
    close(dev("expm1", x), np.expm1(x.astype(L)), 3 * U)
    for fn in ("artanh", "cosh", "sinhc"):
        assert dev(fn, np.zeros(1))[0] == 1.0
    w = spread(8, -3, 3)
    for n in range(1, 9):
        close(dev("power", w, np.full_like(w, n)), w.astype(L) ** n, 8 * U)


def test_conversions_give_the_bits_of_the_instructions(dev):
    with np.errstate(all="ignore"):
        rng = np.random.default_rng(9)
        f = np.concatenate([rng.integers(0, 2 ** 32, 400000, dtype=np.uint64).astype(np.uint32),
                            np.array([0, 1, 0x7fffff, 0x800000, 0x7f7fffff, 0x7f800000], np.uint32)])
        f = np.concatenate([f, f ^ np.uint32(0x80000000)])
        same(dev("widen", f.astype(np.uint64).view(np.float64)), f.view(np.float32).astype(np.float64))
        # halfway between neighbours of FP32, even and odd, and one unit to each side; then every exponent
        base = np.concatenate([rng.integers(0x00800000, 0x7f7fffff, 100000),
                               [0x7f7fffff, 0x00800000, 0, 1, 2, 0x3f800000]])
        base = base.astype(np.uint32).view(np.float32).astype(np.float64)
        half = base + np.abs(np.spacing(base.astype(np.float32)).astype(np.float64)) / 2
        x = np.concatenate([base, half, np.nextafter(half, 0), np.nextafter(half, INF), spread(10, -1074, 1023),
                            spread(11, -160, 130), EDGES, [NAN]])
        x = np.concatenate([x, -x])
        got = dev("narrow", x).view(np.uint64).astype(np.uint32).view(np.float32)
        want = x.astype(np.float32)
        ok = (got.view(np.uint32) == want.view(np.uint32)) | (np.isnan(got) & np.isnan(want))
        assert np.all(ok), x[~ok][:4]


def test_comparisons_give_the_values_of_the_operators(dev):
    with np.errstate(all="ignore"):
        e = np.concatenate([EDGES, -EDGES, [NAN], spread(12, -1074, 1023, 60), spread(13, -1, 1, 60)])
        a, b = [m.ravel() for m in np.meshgrid(e, e)]
        p = (a > 0) + 2.0 * (a < 0) + 4.0 * (a >= 0) + 8.0 * (a == 0) + 16.0 * (a > 1)
        same(dev("pred", a), p)
        ok = ~(np.isnan(a) | np.isnan(b)) & ~((a == 0) & (b == 0))     # of numbers; zeros of either sign have an order
        same(dev("less", a[ok], b[ok]), (a < b)[ok].astype(float))
        for name, fn in (("min", np.fmin), ("max", np.fmax)):
            got, want = dev(name, a, b), fn(a, b)
            assert np.all((got == want) | (np.isnan(got) & np.isnan(want)))


@pytest.mark.parametrize("yield_strain", [1e-3, 1e-5, 4e-7])
def test_fp32_cells_beyond_a_small_yield_strain_yield(lib, yield_strain):
    """Stretches of 0.8 to 1.3 times the yield strain, exact in FP32, in the FP32
    form: the plastic strain is that of the FP64 return (its factor 1 - s by the
    FP32 rounding of G, 1e-7; allowed 1e-6 of |dev H|), none below yield."""
    n, G0, rho0 = 20000, 26e9, 2700.0
    rng = np.random.default_rng(14)
    d = rng.standard_normal((5, n))
    d[4] = -(d[0] + d[3])
    d *= yield_strain * rng.uniform(0.8, 1.3, n) / np.sqrt(d[0] ** 2 + d[3] ** 2 + d[4] ** 2 + (d[1] + d[2]) ** 2 / 2)
    A = np.ascontiguousarray(d + np.array([1, 0, 0, 1, 1])[:, None], dtype=np.float32)
    a = A.astype(np.longdouble)
    # |dev ln V| by the eigenvalues of the in-plane block of A A^T less 1
    b00 = (a[0] - 1) * (a[0] + 1) + a[1] ** 2
    b11 = (a[3] - 1) * (a[3] + 1) + a[2] ** 2
    b01 = a[0] * a[2] + a[1] * a[3]
    mid, rad = (b00 + b11) / 2, np.sqrt(((b00 - b11) / 2) ** 2 + b01 ** 2)
    h = np.array([np.log1p(mid + rad), np.log1p(mid - rad), np.log1p((a[4] - 1) * (a[4] + 1))]) / 2
    norm = np.sqrt(((h - h.mean(axis=0)) ** 2).sum(axis=0))
    sig_y = np.sqrt(6.0) * G0 * yield_strain
    want = np.sqrt(np.longdouble(2) / 3) * np.maximum(norm - yield_strain, 0)
    strain = np.empty(n, dtype=np.float32)
    fp = ctypes.POINTER(ctypes.c_float)
    lib.dm_finish.argtypes = [ctypes.c_double] * 4 + [fp, fp, ctypes.c_int]
    assert lib.dm_finish(rho0, 76e9, G0, sig_y, A.ctypes.data_as(fp), strain.ctypes.data_as(fp), n) == 0
    assert np.any(want > 0) and np.any(want == 0)
    assert np.all(np.abs(strain / rho0 - want) <= 1e-6 * norm)
