"""Scalar device functions of the library (tests/device_functions.cu, compiled
here with the library's flags) against exact values."""
import ctypes
import os
from decimal import Decimal, localcontext

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
