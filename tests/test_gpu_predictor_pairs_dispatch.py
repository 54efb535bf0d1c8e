"""Every node-pair form that the per-mesh mixed step chooses by its number of
cells (degrees 3, 5, 7; uniform cells and the leaves of adaptive meshes)
against the node-per-thread body of the batched launch, bitwise: with exactly
the largest number of cells of one form and just above it, the last block of
the next form ragged.  The numbers of cells follow the device's SM count."""
import pytest
import torch

from paper_1905_05524_gb300 import _lib as L
from paper_1905_05524_gb300.solver import Batch, Mesh, atmosphere_config

pytestmark = pytest.mark.gpu

# degree, cells per SM up to which a form runs, cells per block of the form above
BOUNDS = [(3, 64, 16), (5, 12, 7), (7, 4, 1), (7, 8, 2)]


def _mesh(degree, nx, ny, refine=()):
    cfg = atmosphere_config(degree=degree, nx=nx, ny=ny, precision=L.ADG_PREC_MIXED)
    cfg.max_levels = 1 if refine else 0
    m = Mesh(cfg)
    m.init_scenario(L.ADG_SCEN_COSINE, A=0.5, a=250.0, xc=500.0, zc=350.0)
    if refine:
        fl = torch.zeros(nx * ny, dtype=torch.int8)
        fl[list(refine)] = 1
        m.adapt(fl.cuda())
        assert m.leaves > nx * ny
    u = m.get_state()
    g = torch.Generator(device="cuda").manual_seed(degree)
    r = torch.rand(u[:, 1:3].shape, generator=g, dtype=torch.float64, device="cuda") - 0.5
    u[:, 1:3] += 0.5 * r * u[:, 0:1]  # momentum everywhere: every flux term is active
    m.set_state(u)
    return m


def _check(make):
    a, b = make(), make()
    dt = a.stable_dt(0.25)
    batch = Batch([b])
    batch.set_candidate(1)
    a.step(dt, 2)
    batch.step([dt], 2)
    torch.cuda.synchronize()
    assert torch.isfinite(a.get_state()).all()
    assert torch.equal(a.get_state(), b.get_state())
    batch.close()
    a.close()
    b.close()


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _above(limit, cpb, more=0):
    """Columns of a mesh three cells high with a few cells above the limit, with `more` not a multiple of cpb."""
    nx = limit // 3 + 1
    while cpb > 1 and (3 * nx + more) % cpb == 0:
        nx += 1
    return nx


@pytest.mark.parametrize("degree,per_sm,cpb", BOUNDS)
def test_uniform_at_and_above_each_bound(degree, per_sm, cpb):
    sms = _sms()
    _check(lambda: _mesh(degree, sms, per_sm))
    _check(lambda: _mesh(degree, _above(per_sm * sms, cpb), 3))


@pytest.mark.parametrize("degree,per_sm,cpb", BOUNDS)
def test_adaptive_above_each_bound(degree, per_sm, cpb):
    """Refined leaves at a corner, on a wall and inside: hanging faces beside walls and cells."""
    nx = _above(per_sm * _sms(), cpb, 5 * 8)
    _check(lambda: _mesh(degree, nx, 3, refine=(0, 1, nx // 2, nx + nx // 2, 2 * nx + 5)))
