"""Fixed-point contractions of the FP64 path (csrc/adg_fixed.cuh).

On the host, an integer model of the arithmetic against exact rationals: a dot
product of n <= 8 doubles (16 for the divergence's two rows) with common
exponents taken from the largest magnitudes.  Truncating each operand to 58
bits moves it by less than 2^-57 of the group's largest (the group's power of
two is at most twice that), the dropped low-by-low products are below 2^-57 of
max|a| max|b| per term and the combination rounds once, so the error stays
below (3 n + 1) 2^-57 max|a| max|b|; the result rounds to a double.

On the GPU: multiplying rho, rho v, rho E and mu by a power of two scales every
term of the equations by it, and every operation of the step is exact under
that scaling, so the step must scale bitwise; a NaN stays in its cell and the
face neighbours.
"""
import math
import struct
from fractions import Fraction

import numpy as np
import pytest
import torch


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _exp(xs):
    return max(max((_bits(x) >> 52) & 0x7FF for x in xs), 256)


def _from(x, E):
    b = _bits(x)
    t = (((b & ((1 << 52) - 1)) | 1 << 52) << 5) >> min(E - ((b >> 52) & 0x7FF), 63)
    return -t if b >> 63 else t


def _dot(a, b):
    """Integer value and binary exponent of the dot product, as the kernel forms it."""
    Ea, Eb = _exp(a), _exp(b)
    hh = mid = 0
    for x, y in zip(a, b):
        m, q = _from(x, Ea), _from(y, Eb)
        ah = (m + (1 << 28)) >> 29
        al = m - (ah << 29)
        bh, bl = q >> 29, q & 0x1FFFFFFF
        assert abs(ah) <= 1 << 29 and abs(al) <= 1 << 28 and abs(bh) <= 1 << 29
        hh += ah * bh
        mid += ah * bl + al * bh
        assert abs(hh) < 1 << 63 and abs(mid) < (1 << 63) - (1 << 28)
    return hh + ((mid + (1 << 28)) >> 29), Ea + Eb - 2102


@pytest.mark.parametrize("n", [2, 3, 6, 8, 16])
@pytest.mark.parametrize("spread", [0, 40, 400])
def test_dot_product_error_bound(n, spread):
    rng = np.random.default_rng(100 * n + spread)
    for _ in range(300):
        a = [float(x) for x in rng.uniform(-1, 1, n) * 2.0 ** rng.uniform(-min(spread, 4), 0, n) * 2.0 ** rng.integers(-30, 30)]
        b = [float(x) for x in rng.uniform(-1, 1, n) * 2.0 ** rng.uniform(-spread, 0, n) * 2.0 ** rng.integers(-300, 300)]
        if rng.random() < 0.2:
            b[int(rng.integers(n))] = 0.0
        v, e = _dot(a, b)
        got = Fraction(v) * Fraction(2) ** e
        want = sum(Fraction(x) * Fraction(y) for x, y in zip(a, b))
        top = Fraction(max(map(abs, a))) * Fraction(max(map(abs, b)))
        assert abs(got - want) <= (3 * n + 1) * top / 2 ** 57


def test_dot_product_at_the_largest_operands():
    big = math.nextafter(2.0, 1.0)
    for n in (8, 16):
        for s in (1.0, -1.0):
            v, e = _dot([big] * n, [s * big] * n)
            want = n * Fraction(big) ** 2 * int(s)
            assert abs(Fraction(v) * Fraction(2) ** e - want) <= (3 * n + 1) * Fraction(4) / 2 ** 57


# ------------------------------------------------------------------- GPU
def _steady(degree, nx, ny, scale, source):
    from paper_1905_05524_gb300 import _lib as L
    from paper_1905_05524_gb300.solver import Mesh, steady_manufactured_config
    cfg = steady_manufactured_config(degree=degree, nx=nx, ny=ny)
    cfg.mu *= scale
    if not source:
        cfg.source = L.ADG_SRC_NONE
    return cfg, Mesh(cfg)


def _flow(cfg, seed):
    """Random smooth-enough nodal data around a moving gas at rest density 1."""
    n = cfg.degree + 1
    g = torch.Generator().manual_seed(seed)
    r = [torch.rand(cfg.nx * cfg.ny, n, n, generator=g, dtype=torch.float64) - 0.5 for _ in range(4)]
    rho = 1.0 + 0.02 * r[0]
    u, v, p = 0.5 + 0.02 * r[1], -0.3 + 0.02 * r[2], 1.0 + 0.02 * r[3]
    return torch.stack([rho, rho * u, rho * v, p / 0.4 + 0.5 * rho * (u * u + v * v)], 1).contiguous()


@pytest.mark.gpu
@pytest.mark.parametrize("degree,nx,ny", [(1, 3, 2), (2, 5, 1), (3, 2, 3), (4, 1, 3), (5, 3, 3), (6, 2, 1), (7, 1, 2)])
@pytest.mark.parametrize("power", [-180, -1, 7, 180])
def test_step_scales_bitwise_with_powers_of_two(degree, nx, ny, power):
    out = []
    for s in (1.0, 2.0 ** power):
        cfg, m = _steady(degree, nx, ny, s, False)
        m.set_state((_flow(cfg, degree) * s).cuda())
        for _ in range(2):
            m.step(1e-3)
        out.append(m.get_state().cpu())
        m.close()
    assert torch.isfinite(out[0]).all()
    assert torch.equal(out[0] * 2.0 ** power, out[1])


@pytest.mark.gpu
@pytest.mark.parametrize("degree", [1, 3, 5, 7])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_values_stay_with_the_face_neighbours(degree, bad):
    got = []
    for plant in (False, True):
        cfg, m = _steady(degree, 5, 5, 1.0, True)
        u = _flow(cfg, 9)
        if plant:
            u[12, 3, 0, degree] = bad
        m.set_state(u.cuda())
        m.step(1e-3)
        got.append(m.get_state().cpu())
        m.close()
    hit = {12, 11, 13, 7, 17}
    for c in range(25):
        if c in hit:
            assert not torch.isfinite(got[1][c]).all()
        else:
            assert torch.equal(got[0][c], got[1][c])
