"""Scalar device functions of the library (tests/device_functions.cu, compiled
here with the library's flags) against exact values."""
import ctypes
import math
import os
from decimal import Decimal, localcontext
from fractions import Fraction

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    from paper_1905_05524_gb300 import build as b
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_functions.cu")
    so = str(tmp_path_factory.mktemp("dev") / "device_functions.so")
    b._run([b._nvcc(), *b.ARCH, *b.FLAGS, "-I", b.CSRC, "-shared", "-o", so, src])
    torch.cuda.init()
    return ctypes.CDLL(so)


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("lo,hi", [(0.88, 1.02), (0.6, 1.65), (0.3, 3.0)])
def test_theta_is_as_accurate_as_pow(dev, lo, hi):
    """theta = T (p0/p)^(R/cp) in the lowest kilometre, over the range of the
    exp/log form and on both sides of its ends: its error, in units of 2^-53 of
    theta, against 40 digits is no larger than that of T pow(p0/p, R/cp)."""
    p0, Rcp, n = 1e5, 2.0 / 7.0, 20000
    p = np.random.default_rng(7).uniform(lo * p0, hi * p0, n)
    x = torch.from_numpy(p).cuda()
    out = torch.empty(2, n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert dev.dev_theta(_p(x), _p(out), n, ctypes.c_double(p0), ctypes.c_double(Rcp)) == 0
    got = out.cpu().numpy()
    with localcontext() as c:
        c.prec = 40
        want = [Decimal(v) * (Decimal(Rcp) * (Decimal(p0) / Decimal(v)).ln()).exp() for v in p.tolist()]
        err = np.array([[float((Decimal(g) - w) / w) for g, w in zip(row.tolist(), want)] for row in got]) * 2.0 ** 53
    rms, top = np.sqrt((err ** 2).mean(1)), np.abs(err).max(1)
    print(f"rms {rms}, largest {top}")
    assert rms[0] <= rms[1] and top[0] <= top[1]


def test_3d_mixed_flux_divides_by_the_density_correctly_rounded(dev):
    """1/rho of the 3D mixed flux (rho u v with both momenta 1) is the nearest
    float, over the densities of gases and far from them."""
    rng = np.random.default_rng(3)
    rho = np.concatenate([rng.uniform(0.5, 1.5, 20000), 2.0 ** rng.uniform(-120, 120, 20000)]).astype(np.float32)
    x = torch.from_numpy(rho).cuda()
    out = torch.empty_like(x)
    torch.cuda.synchronize()
    assert dev.dev_flux3_rcp(_p(x), _p(out), rho.size) == 0
    # 1/rho in 64 bits rounds to the nearest float unless it lies within 2^-53 of a tie, which 24-bit rho rule out
    assert np.array_equal(out.cpu().numpy(), (1.0 / rho.astype(np.float64)).astype(np.float32))


def _doubles(rng, exps):
    """Doubles of the given biased exponents with random and edge mantissas, both signs."""
    e = np.repeat(np.asarray(exps, dtype=np.uint64), 8)
    m = rng.integers(0, 1 << 52, e.size, dtype=np.uint64)
    edge = np.array([0, 1, (1 << 52) - 1, 1 << 51, (1 << 29) - 1, 1 << 29], dtype=np.uint64)
    k = np.arange(e.size) % 8
    m = np.where(k < 6, edge[np.minimum(k, 5)], m)
    s = rng.integers(0, 2, e.size, dtype=np.uint64)
    return (s << np.uint64(63) | e << np.uint64(52) | m).view(np.float64)


def test_reciprocal(dev):
    """One Newton-like step of third order from 2^-22 leaves 2^-66, so the result
    is within (1/2 + 2^-12) of its last place; subnormal, huge and special values
    take the division."""
    rng = np.random.default_rng(5)
    x = np.concatenate([_doubles(rng, np.arange(2047)), [0.0, -0.0, np.inf, -np.inf, np.nan], rng.uniform(0.5, 2.0, 20000)])
    t = torch.from_numpy(x).cuda()
    out = torch.empty_like(t)
    torch.cuda.synchronize()
    assert dev.dev_rcp(_p(t), _p(out), x.size) == 0
    got = out.cpu().numpy()
    with np.errstate(divide="ignore", over="ignore"):
        div = 1.0 / x
    ex = (x.view(np.uint64) >> np.uint64(52) & np.uint64(0x7FF)).astype(int)
    far = (ex == 0) | (ex > 2040)
    assert np.array_equal(got[far], div[far], equal_nan=True)
    for a, r in zip(x[~far].tolist(), got[~far].tolist()):
        fr = Fraction(r)
        assert abs(fr - 1 / Fraction(a)) <= (Fraction(1, 2) + Fraction(1, 4096)) * Fraction(math.ulp(r))


def test_fixed_point_from_double(dev):
    """m = x 2^(1080 - E) cut to an integer below 2^58, and both splits of it."""
    rng = np.random.default_rng(6)
    x = _doubles(rng, np.concatenate([[0], np.arange(200, 2047, 3)]))
    ex = (x.view(np.uint64) >> np.uint64(52) & np.uint64(0x7FF)).astype(int)
    E = np.maximum(ex + rng.choice([0, 1, 2, 5, 30, 57, 58, 63, 300], x.size), 256).astype(np.int32)
    tx, tE = torch.from_numpy(x).cuda(), torch.from_numpy(E).cuda()
    m = torch.empty(x.size, dtype=torch.int64, device="cuda")
    limbs = torch.empty(x.size, 4, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert dev.dev_from(_p(tx), _p(tE), _p(m), _p(limbs), x.size) == 0
    for a, e, k, (h, l, ch, cl) in zip(x.tolist(), E.tolist(), m.cpu().tolist(), limbs.cpu().tolist()):
        want = abs(Fraction(a)) * Fraction(2) ** (1080 - e) if abs(a) >= 2.0 ** -1022 else 0
        assert abs(k) == int(want) < 1 << 58 and (k == 0 or (k < 0) == (a < 0))
        assert h * (1 << 29) + l == k and 0 <= l < 1 << 29
        assert ch * (1 << 29) + cl == k and abs(cl) <= 1 << 28 and abs(ch) <= 1 << 29


def test_double_from_fixed_point(dev):
    """a 2^e rounds to the nearest double, ties away from zero; NaN above the
    range, zero below the normal numbers."""
    rng = np.random.default_rng(8)
    bits = np.tile(np.arange(1, 63), 60)
    a = np.array([int(rng.integers(1 << (b - 1), 1 << b)) for b in bits.tolist()])
    pat = np.arange(a.size) % 6
    a = np.where(pat == 0, 1 << (bits - 1), np.where(pat == 1, (1 << bits) - 1, a))
    a = np.where(rng.random(a.size) < 0.5, -a, a)
    e = rng.integers(-1100, 1050, a.size).astype(np.int32)
    a, e = np.append(a, [0, 0]), np.append(e, [0, 30000]).astype(np.int32)
    ta, te = torch.from_numpy(a).cuda(), torch.from_numpy(e).cuda()
    out = torch.empty(a.size, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert dev.dev_to(_p(ta), _p(te), _p(out), a.size) == 0
    for m, x, r in zip(a.tolist(), e.tolist(), out.cpu().tolist()):
        top = abs(m).bit_length() + x  # |a 2^e| in [2^(top - 1), 2^top)
        if (m == 0 and x < 2046) or (m and top - 1 < -1022):
            assert r == 0.0
        elif m == 0 or top > 1024:
            assert math.isnan(r)
        else:
            cut = max(abs(m).bit_length() - 53, 0)
            mag = (abs(m) + (1 << cut >> 1)) >> cut
            want = Fraction(mag) * Fraction(2) ** (x + cut) * (1 if m > 0 else -1)
            assert Fraction(r) == want if want < Fraction(2) ** 1024 else math.isinf(r)
