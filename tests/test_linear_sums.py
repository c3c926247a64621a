"""The float64 step's lattice sums in block fixed point, on arrays: exact
rational arithmetic against the host build of the functions (CPU), the device
against the host bit for bit (GPU)."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2508_16997_gb300 import build

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = [Fraction(4, 9)] + [Fraction(1, 9)] * 4 + [Fraction(1, 36)] * 4
T = Fraction(1, 3)

# rows of integers: the sums' coefficients per input
MOMENTS = [[1] * 9, list(EX), list(EY),
           [3 * x * x - 1 for x in EX], [3 * y * y - 1 for y in EY],
           [x * y for x, y in zip(EX, EY)],
           [(3 * x * x - 1) * y for x, y in zip(EX, EY)],
           [(3 * y * y - 1) * x for x, y in zip(EX, EY)]]
# inputs b0/9, bx/3, by/3, bxx/3, byy/3, bxy, bxxy, bxyy
POPULATIONS = [[w * 9, w * 3 * x * 3, w * 3 * y * 3, w * Fraction(9, 2) * (x * x - T) * 3,
                w * Fraction(9, 2) * (y * y - T) * 3, w * 9 * x * y,
                w * Fraction(27, 2) * (x * x - T) * y, w * Fraction(27, 2) * (y * y - T) * x]
               for w, x, y in zip(W, EX, EY)]


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    here = os.path.dirname(os.path.abspath(__file__))
    so = str(tmp_path_factory.mktemp("probe") / "linear_probe.so")
    cmd = [build.nvcc(), *build.NVCC_FLAGS, f"-I{build.CSRC}", "-shared", "-o", so,
           os.path.join(here, "linear_probe.cu")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


@pytest.fixture()
def gpu_probe(probe):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return probe


def _ptr(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


def sums(fn, kind, third, a):
    a = np.ascontiguousarray(a, dtype=np.float64)
    out = np.empty((len(a), 8 if kind == 0 else 9))
    rc = fn(kind, int(third), _ptr(a), _ptr(out), ctypes.c_longlong(len(a)))
    assert fn.__name__.endswith("host") or rc == 0
    return out


def inputs(kind, third, n, seed):
    """Rows over many binades: equal sizes, one large value, spread exponents,
    zeros, ties."""
    rng = np.random.default_rng(seed)
    m = 9 if kind == 0 else 8
    a = rng.uniform(-1, 1, (n, m))
    a *= 2.0 ** rng.integers(-1, 1, (n, m))
    spread = rng.choice([0, 3, 8, 20, 45, 60, 70], n)[:, None]
    a *= 2.0 ** -(rng.integers(0, 1000, (n, m)) % (spread + 1))
    a *= 2.0 ** rng.choice([0, -40, 300, -800, 900], n)[:, None].astype(float)
    a[rng.random((n, m)) < 0.1] = 0.0
    short = rng.random((n, m)) < 0.2  # values of four bits: ties
    frac, e = np.frexp(a)
    a = np.where(short, np.ldexp(np.round(frac * 16) / 16, e), a)
    if kind == 1 and not third:
        a[:, 6:] = 0.0
    return a


def exponent(v):
    """Biased exponent field of float64 values."""
    return (np.asarray(v, dtype=np.float64).view(np.uint64) >> np.uint64(52)).astype(int) & 0x7ff


def unit_of(row):
    """Last place of a row's block: the largest value's leading bit is bit 58."""
    return Fraction(2) ** (max(64, int(exponent(row).max())) - 1023 - 58)


def half_ulp(v):
    return Fraction(float(np.spacing(abs(v)))) / 2


@pytest.mark.parametrize("kind,third", [(0, True), (0, False), (1, True), (1, False)])
def test_sums_within_their_roundings(probe, kind, third):
    """Every result within half an ulp of the exact sum plus, for each operand
    with bits below the block's last place, half of that place."""
    a = inputs(kind, third, 3000, 1)
    out = sums(probe.probe_sums_host, kind, third, a)
    half = Fraction(1, 2)
    for row, got in zip(a, out):
        x = [Fraction(v) for v in row]
        unit = unit_of(row)
        loose = [(v / unit).denominator != 1 for v in x]
        rows = MOMENTS if kind == 0 else POPULATIONS
        for j, c in enumerate(rows):
            if kind == 0 and j >= 6 and not third:
                continue
            exact = sum(ci * xi for ci, xi in zip(c, x))
            tol = half_ulp(got[j]) + unit * half * sum(abs(ci) for ci, l in zip(c, loose) if l)
            assert abs(Fraction(got[j]) - exact) <= tol, (row, j)


@pytest.mark.parametrize("bits", [6, 7, 8, 9, 10, 15, 25, 37])
def test_small_operand_keeps_its_mean(probe, bits):
    """The rest population beside two opposite ones 2^bits larger: drho is the rest
    population alone, rounded to nearest, ties away from zero.  20,000 one-signed
    values: apart from 6 standard errors (an error within half a unit has one of at
    most 0.5 / sqrt(n)) the mean rounding is that of the ties, half a unit in one
    of 2^dropped values: half a last place of the operand itself."""
    n = 20000
    rng = np.random.default_rng(bits)
    a = np.zeros((n, 9))
    big = rng.uniform(0.5, 1.0, n)
    a[:, 1], a[:, 3] = big, -big
    # every last bit equally likely (rng.uniform(0.5, 1.0) prefers even ones)
    a[:, 0] = np.ldexp(2.0 ** 52 + rng.integers(0, 2 ** 52, n), -53 - bits)
    drho = sums(probe.probe_sums_host, 0, True, a)[:, 0]
    # the difference of two values of nearly the same size is exact
    err = np.ldexp(drho - a[:, 0], 59)  # in units: the block's exponent is that of 1/2
    assert np.abs(err).max() <= 0.5
    assert abs(err.mean()) <= 0.5 * np.spacing(a[:, 0]).mean() * 2.0 ** 59 + 3 / np.sqrt(n)


def test_ties_go_away_from_zero(probe):
    """k + 1/2 units beside a block of exponent 0, of either sign."""
    k = np.arange(0, 64)
    for sign in (1.0, -1.0):
        a = np.zeros((k.size, 9))
        a[:, 1], a[:, 3] = 1.5, -1.5
        a[:, 0] = sign * np.ldexp(k + 0.5, -58)
        drho = sums(probe.probe_sums_host, 0, True, a)[:, 0]
        np.testing.assert_array_equal(drho, sign * np.ldexp(k + 1.0, -58))


def edge_rows(kind):
    """Zeros, infinities, NaN, subnormals, the ends of the exponent range."""
    m = 9 if kind == 0 else 8
    big, small = np.ldexp(1.0, 1019), np.ldexp(1.0, -1017)
    vals = [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -2.5e-310, np.finfo(float).tiny, small,
            -1.5 * small, 0.75 * small, big, -1.9999 * big, np.ldexp(1.0, 1020),
            np.finfo(float).max, 1.0, -1.0]
    rows = [np.zeros(m)]
    for v in vals:
        for j in range(m):
            for fill in (0.0, 1.0, small, -big):
                r = np.full(m, fill)
                r[j] = v
                rows.append(r)
        rows.append(np.full(m, v))
    return np.array(rows)


@pytest.mark.parametrize("kind", [0, 1])
def test_edges_of_the_range(probe, kind):
    a = edge_rows(kind)
    out = sums(probe.probe_sums_host, kind, True, a)
    top = exponent(a).max(axis=1)
    assert np.isnan(out[top >= 1023 + 1020]).all()
    assert np.isfinite(out[top < 1023 + 1020]).all()
    assert not out[np.all(a == 0.0, axis=1)].any()
    half = Fraction(1, 2)
    rows = MOMENTS if kind == 0 else POPULATIONS
    for row, got in zip(a[top < 1023 + 1020], out[top < 1023 + 1020]):
        x = [Fraction(v) for v in row]
        for j, c in enumerate(rows):
            exact = sum(ci * xi for ci, xi in zip(c, x))
            tol = half_ulp(got[j]) + unit_of(row) * half * sum(abs(ci) for ci in c)
            assert abs(Fraction(got[j]) - exact) <= tol, (row, j)


@pytest.mark.gpu
@pytest.mark.parametrize("kind,third", [(0, True), (0, False), (1, True), (1, False)])
def test_device_equals_host(gpu_probe, kind, third):
    a = np.concatenate([inputs(kind, third, 20000, 2), edge_rows(kind)])
    host = sums(gpu_probe.probe_sums_host, kind, third, a)
    dev = sums(gpu_probe.probe_sums_device, kind, third, a)
    np.testing.assert_array_equal(dev, host)  # NaN equals NaN
    np.testing.assert_array_equal(np.signbit(dev[dev == 0]), np.signbit(host[host == 0]))


@pytest.mark.gpu
def test_reciprocal(gpu_probe):
    """1 / v: within 1/2 + 2^-12 units of the last place over [2^-100, 2^101), the
    division itself outside.  x has at most 2^-22 relative error (v truncated to
    24 bits, rcp.approx within 2^-23), so the cubic step leaves 2^-66, its two
    inner roundings 2^-75 each: together below 2^-13 units before the last
    rounding."""
    rng = np.random.default_rng(5)
    n = 200000
    near = np.concatenate([1.0 + rng.uniform(-0.1, 0.1, n // 2), rng.uniform(1.0, 2.0, n // 2)])
    wide = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-100, 101, n))
    edges = np.array([np.nextafter(np.ldexp(1.0, k), s) for k in range(-100, 101)
                      for s in (0.0, np.inf)] + [np.ldexp(1.0, k) for k in range(-100, 101)])
    edges = edges[(edges >= 2.0 ** -100) & (edges < 2.0 ** 101)]
    v = np.concatenate([near, wide, edges])
    v[::3] *= -1.0
    out = np.empty_like(v)
    assert gpu_probe.probe_recip_device(_ptr(v), _ptr(out), ctypes.c_longlong(v.size)) == 0
    # exact in integers: |out v - 1| against ulp(out) v / 2 (1 + 2^-11), every 7th value
    for a, r in zip(v[::7], out[::7]):
        exact = 1 / Fraction(a)
        assert abs(Fraction(r) - exact) <= Fraction(float(np.spacing(abs(r)))) * (
            Fraction(1, 2) + Fraction(1, 2 ** 12)), a
    # all of them against the correctly rounded quotient: at most one place off
    assert (np.abs(out - 1.0 / v) <= np.spacing(np.abs(out))).all()

    v = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310, np.finfo(float).tiny,
                  np.finfo(float).max, np.ldexp(1.0, 101), -np.ldexp(1.5, 300),
                  np.nextafter(2.0 ** -100, 0.0), -np.ldexp(1.1, -500)])
    out = np.empty_like(v)
    assert gpu_probe.probe_recip_device(_ptr(v), _ptr(out), ctypes.c_longlong(v.size)) == 0
    with np.errstate(divide="ignore", over="ignore"):
        np.testing.assert_array_equal(out, 1.0 / v)
