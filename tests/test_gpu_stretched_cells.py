"""Cells 2^24 times longer along one axis (l) than along the other (s): the FP64
step and its adjoint keep the derivatives along the long side to their own
accuracy, not to that of the short side's (2^24 times larger) entries of D / h.

A flow along s, v_s = f(x_s) g(x_l), over uniform density and pressure leaves
the momentum along l to the viscous stress alone (it starts at zero):
    d m_l / dt = d_s(mu d_l v_s) - d_l(2/3 mu d_s v_s),
one derivative along each axis.  Each of the 2 n + 16 roundings between the
state and a value of d m_l is at most eps = 2^-52 of the operands' magnitudes:
with L the largest row or column sum of |D|, W that of the weak volume term and
of the lifting, per unit cell length, the two operands of each gradient
(d(rho v) and v d(rho)) give (2 + 4/3) mu U L W / (h_l h_s), the pressure, which
the long derivative of the normal flux cancels, p W / h_l.  Two implementations
differ by at most twice that.  The adjoint is the transpose: an adjoint of m_l
alone gives one of m_s, with (gamma - 1) U for p.
"""
import numpy as np
import pytest
import torch

from oracle.basis import Basis
from paper_1905_05524_gb300.solver import Mesh, Mesh3, Mesh3Config, MeshConfig
from tests.oracle_bridge import oracle_for
from tests.test_gpu_3d import oracle3
from tests.test_gpu_adjoint import gpu_adjoint, oracle_adjoint

pytestmark = pytest.mark.gpu

LONG, MU, DT = 2.0 ** 24, 1.0, 2.0 ** -30


def bound(degree, inertia):
    B = Basis(degree)
    n = degree + 1
    D, w = np.asarray(B.D, dtype=float), np.asarray(B.w, dtype=float)
    phi = [np.abs(np.asarray(p, dtype=float)) for p in (B.phi0, B.phi1)]
    V = np.abs(w[:, None] * D / w[None, :])
    L = max(np.abs(D).sum(0).max(), np.abs(D).sum(1).max())
    W = max(V.sum(0).max(), V.sum(1).max()) + 2.0 * max(p.max() * (p / w).sum() for p in phi)
    return 2.0 * DT * 2.0 ** -52 * (2 * n + 16) * W / LONG * (10.0 / 3.0 * MU * 1.5 * L + inertia)


def flow(X, l, s, H, dims):
    """v_s = f(x_s) g(x_l), rho = p = 1 (|v_s| <= 1.5)."""
    x = [X[a] * (2.0 * np.pi / (2.0 * H[a])) for a in range(dims)]
    v = (0.9 + 0.3 * torch.sin(x[s] + 0.3)) * (0.9 + 0.3 * torch.cos(x[l] - 0.4))
    one = torch.ones_like(v)
    m = [0.0 * one] * dims
    m[s] = v
    return torch.stack([one, *m, one / 0.4 + 0.5 * v * v], 1)


def check(got, want, tol):
    err, size = (got - want).abs().max().item(), want.abs().max().item()
    assert size > 100.0 * tol, (size, tol)
    assert err <= tol, (err, tol, size)


@pytest.mark.parametrize("long", [0, 1])
@pytest.mark.parametrize("degree", [1, 2, 3, 5, 7])
def test_step_2d(degree, long):
    H = [1.0, 1.0]
    H[long] = LONG
    cfg = MeshConfig(degree=degree, nx=2, ny=2, Lx=2.0 * H[0], Ly=2.0 * H[1], mu=MU)
    o = oracle_for(cfg)
    u0 = flow((o.X, o.Y), long, 1 - long, H, 2)
    m = Mesh(cfg)
    m.set_state(u0.cuda().contiguous())
    m.step(DT)
    check(m.get_state().cpu()[:, 1 + long], o.step(u0, DT)[:, 1 + long], bound(degree, 1.0))
    m.close()


@pytest.mark.parametrize("long", [0, 1, 2])
@pytest.mark.parametrize("degree", [1, 2, 3, 4])
def test_step_3d(degree, long):
    H = [1.0, 1.0, 1.0]
    H[long] = LONG
    cfg = Mesh3Config(degree=degree, nx=2, ny=2, nz=2, Lx=2.0 * H[0], Ly=2.0 * H[1], Lz=2.0 * H[2], mu=MU)
    o = oracle3(cfg)
    u0 = flow((o.X, o.Y, o.Z), long, (long + 1) % 3, H, 3)
    m = Mesh3(cfg)
    m.set_state(u0)
    m.step(DT)
    check(m.get_state().cpu()[:, 1 + long], o.step(u0, DT)[:, 1 + long], bound(degree, 1.0))
    m.close()


@pytest.mark.parametrize("long", [0, 1])
@pytest.mark.parametrize("degree", [1, 2, 3, 4, 5])
def test_adjoint_2d(degree, long):
    H = [1.0, 1.0]
    H[long] = LONG
    cfg = MeshConfig(degree=degree, nx=2, ny=2, Lx=2.0 * H[0], Ly=2.0 * H[1], mu=MU)
    o = oracle_for(cfg)
    u0 = flow((o.X, o.Y), long, 1 - long, H, 2)
    lam = torch.zeros_like(u0)
    lam[:, 1 + long] = 2.0 * torch.rand(lam[:, 0].shape, generator=torch.Generator().manual_seed(degree),
                                        dtype=torch.float64) - 1.0
    m = Mesh(cfg)
    got = gpu_adjoint(m, DT, u0.cuda().contiguous(), lam.cuda().contiguous()).cpu()
    check(got[:, 2 - long], oracle_adjoint(o, DT, u0, lam)[:, 2 - long], bound(degree, 0.4 * 1.5))
    m.close()
