"""The arithmetic that replaces instructions in every solver: the inline division against the exact quotient
and CUDA's, the exact conversion of floats, and the fixed-point sum against exact sums.

Bounds. quotient: the reciprocal estimate's error is cubed and the quotient corrected by its residual, whose
own error is below 2^-50 units in the last place: half a unit plus 2^-50. warp_sum_fixed: each addend is cut
below 2^-62 of the power of two at the largest, and the total is rounded once: addends x 2^-61 of the
largest, plus half a unit."""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_12105_gb300 import build
    so = str(tmp_path_factory.mktemp("device_functions") / "libdevice_functions.so")
    subprocess.run([build.nvcc_path(), *build.ARCH, *build.NVCC_FLAGS, "-shared", "-cudart=shared", "-o", so,
                    os.path.join(HERE, "device_functions.cu")], check=True, capture_output=True, text=True)
    torch.zeros(1, device=DEV)  # the CUDA context
    return ctypes.CDLL(so)


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _quotient(lib, a, b):
    ta, tb = (torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in (a, b))
    q, d = torch.empty_like(ta), torch.empty_like(ta)
    torch.cuda.synchronize()
    assert lib.df_quotient(_p(ta), _p(tb), _p(q), _p(d), ta.numel()) == 0
    return q.cpu().numpy(), d.cpu().numpy()


def _random(rng, n, lo, hi):
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    e = rng.integers(1023 + lo, 1023 + hi, n).astype(np.uint64)
    s = rng.integers(0, 2, n).astype(np.uint64)
    return (s << np.uint64(63) | e << np.uint64(52) | m).view(np.float64)


def test_quotient_of_ordinary_operands(lib):
    """Random mantissas over the whole range of the inline form: the division's own bits (a quotient within
    2^-50 units of a rounding boundary would be allowed to differ; one in 2^49 is)."""
    rng = np.random.default_rng(1)
    for lo, hi in ((-2, 2), (-60, 60), (-399, 400)):
        a, b = _random(rng, 1 << 22, lo, hi), _random(rng, 1 << 22, lo, hi)
        q, d = _quotient(lib, a, b)
        assert np.array_equal(q.view(np.uint64), d.view(np.uint64))


def test_quotient_next_to_rounding_boundaries(lib):
    """a / b at a distance of 1 / (b 2^54) from a midpoint of two doubles, the least there is: within
    half a unit and 2^-50 of the exact quotient."""
    rng = np.random.default_rng(2)
    a, b = [], []
    while len(a) < 4000:
        ib = int(rng.integers(1 << 52, 1 << 53)) | 1
        for sign in (1, -1):
            m = pow(ib, -1, 1 << 54) * sign % (1 << 54)  # m b = sign (mod 2^54), m odd
            ia = (m * ib - sign) >> 54
            if m >> 53 and ia >> 52 == 1:
                a.append(float(ia))
                b.append(float(ib))
    a, b = np.array(a), np.array(b)
    q, d = _quotient(lib, a, b)
    for x, y, z in zip(a, b, q):
        exact = Fraction(float(x)) / Fraction(float(y))
        unit = Fraction(float(np.spacing(float(exact))))
        assert abs(Fraction(float(z)) - exact) <= unit * (Fraction(1, 2) + Fraction(1, 1 << 50))
    assert np.abs(q - d).max() <= np.spacing(np.abs(d)).max()


def test_quotient_falls_back(lib):
    """Around both ends of the inline form's range (exponents of 2^-400 and 2^400) and outside: zeros,
    subnormals, infinities and NaN give the division's bits (any NaN for a NaN); inside, operands like
    1 / (2 - 2^-52) have quotients next to a rounding boundary."""
    rng = np.random.default_rng(3)
    edge = [math.ldexp(1.0, e) for e in (-401, -400, -399, 399, 400, 401, 402, -1022, 1023)]
    special = [0.0, -0.0, 5e-324, -5e-324, 2.0**-1040, np.inf, -np.inf, np.nan, np.finfo(float).max,
               np.finfo(float).tiny, 1.0, -3.0]
    v = np.array([s * (1.0 + f) for s in edge for f in (0.0, 2.0**-52, 1.0 - 2.0**-52)] + special)
    v = np.concatenate([v, -v, _random(rng, 400, -1000, 1000)])
    a, b = (x.reshape(-1).copy() for x in np.meshgrid(v, v))
    q, d = _quotient(lib, a, b)
    nan = np.isnan(d)
    assert np.array_equal(np.isnan(q), nan)
    field = [(x.view(np.uint64) >> np.uint64(52) & np.uint64(0x7ff)).astype(np.int64) for x in (a, b)]
    inline = (np.abs(field[0] - 1023) <= 400) & (np.abs(field[1] - 1023) <= 400)
    differ = ~nan & (q.view(np.uint64) != d.view(np.uint64))
    assert inline.any() and not (differ & ~inline).any()
    for x, y, z in zip(a[differ], b[differ], q[differ]):
        exact = Fraction(float(x)) / Fraction(float(y))
        unit = Fraction(float(np.spacing(abs(float(exact)))))
        assert abs(Fraction(float(z)) - exact) <= unit * (Fraction(1, 2) + Fraction(1, 1 << 50))


def test_widening_is_exact(lib):
    """Every exponent with random and extreme mantissas, both signs, all kinds of denormals, infinities."""
    rng = np.random.default_rng(4)
    e = np.repeat(np.arange(256, dtype=np.uint32), 64)
    m = rng.integers(0, 1 << 23, e.size, dtype=np.uint32)
    m[::64], m[1::64], m[2::64] = 0, (1 << 23) - 1, 1
    u = np.concatenate([e << 23 | m, e << 23 | m | np.uint32(1 << 31), 1 << np.arange(23, dtype=np.uint32)])
    f = u.astype(np.uint32).view(np.float32)
    t, out = torch.from_numpy(f).to(DEV), torch.empty(f.size, dtype=torch.float64, device=DEV)
    torch.cuda.synchronize()
    assert lib.df_widen(_p(t), _p(out), f.size) == 0
    with np.errstate(invalid="ignore"):  # signalling NaN
        want = f.astype(np.float64)
    got = out.cpu().numpy()
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.uint64), want[~nan].view(np.uint64))


def _sums(lib, v, per_lane):
    t = torch.from_numpy(np.ascontiguousarray(v)).to(DEV)
    out = torch.empty((v.shape[0], 32), dtype=torch.float64, device=DEV)
    torch.cuda.synchronize()
    assert lib.df_sum(_p(t), _p(out), v.shape[0], per_lane) == 0
    got = out.cpu().numpy()
    same = got.view(np.uint64) == got[:, :1].view(np.uint64)
    assert (same | np.isnan(got)).all()  # every lane has the sum
    return got[:, 0]


@pytest.mark.parametrize("per_lane", [1, 5])
def test_fixed_point_sums(lib, per_lane):
    """Mixed signs, wide ranges, sums that cancel to nothing or nearly, and both ends of the exponents'
    range (64 above the least; sums that leave the normal numbers)."""
    rng = np.random.default_rng(5)
    n, k = 32 * per_lane, 400
    sets = [rng.uniform(-1, 1, (k, n)), _random(rng, k * n, -60, 60).reshape(k, n), np.abs(rng.standard_normal((k, n))),
            _random(rng, k * n, -1, 1).reshape(k, n) * 2.0**1000, _random(rng, k * n, -3, 3).reshape(k, n) * 2.0**-955]
    x = rng.standard_normal((k, n))
    x[:, n // 2:] = -x[:, :n // 2][:, ::-1]  # cancels exactly
    sets.append(x.copy())
    x[:, 0] += 2.0**-40  # and nearly
    sets += [x, np.zeros((k, n)), np.where(rng.random((k, n)) < 0.9, 0.0, rng.standard_normal((k, n)))]
    for v in sets:
        got = _sums(lib, v, per_lane)
        for row, s in zip(v, got):
            exact = sum((Fraction(float(y)) for y in row), Fraction(0))
            top = float(np.abs(row).max())
            bound = (Fraction(top) * n / (1 << 61) if top else 0) + Fraction(float(np.spacing(abs(float(exact))))) / 2
            assert abs(Fraction(float(s)) - exact) <= bound


@pytest.mark.parametrize("per_lane", [1, 5])
def test_sums_out_of_the_fixed_point_range(lib, per_lane):
    """Tiny addends are added in FP64 (a tree of at most 5 + per_lane roundings); infinities and NaN come through."""
    rng = np.random.default_rng(6)
    n, k = 32 * per_lane, 200
    v = _random(rng, k * n, -40, 1).reshape(k, n) * 2.0**-990
    got = _sums(lib, v, per_lane)
    for row, s in zip(v, got):
        exact = sum((Fraction(float(y)) for y in row), Fraction(0))
        size = sum((abs(Fraction(float(y))) for y in row), Fraction(0))
        assert abs(Fraction(float(s)) - exact) <= size * (5 + per_lane) / (1 << 53) + n * Fraction(5e-324)
    v = rng.standard_normal((6, n))
    v[0, 3] = np.inf
    v[1, n - 1] = -np.inf
    v[2, 0], v[2, n - 1] = np.inf, -np.inf
    v[3, 7] = np.nan
    v[4, :] = np.finfo(float).max
    v[5, :] = -np.finfo(float).max
    got = _sums(lib, v, per_lane)
    assert got[0] == np.inf and got[1] == -np.inf and np.isnan(got[2]) and np.isnan(got[3])
    assert got[4] == np.inf and got[5] == -np.inf
