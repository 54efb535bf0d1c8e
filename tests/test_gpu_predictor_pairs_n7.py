"""The node-pair predictor at degree 7 (two cells per block, padded rows)
against the node-per-thread body of the batched launch: the same operations in
the same order, so bitwise equal, on meshes that end in a full block, in a
half-filled one and in a single cell, with and without walls."""
import pytest
import torch

from paper_1905_05524_gb300 import _lib as L

pytestmark = pytest.mark.gpu


def _mesh(kind, nx, ny, seed):
    from paper_1905_05524_gb300.solver import Mesh, atmosphere_config, steady_manufactured_config
    if kind == "walls":
        m = Mesh(atmosphere_config(degree=7, nx=nx, ny=ny, precision=L.ADG_PREC_MIXED))
        m.init_scenario(L.ADG_SCEN_COSINE, a=300.0)
    else:
        m = Mesh(steady_manufactured_config(degree=7, nx=nx, ny=ny, precision=L.ADG_PREC_MIXED))
        m.init_scenario(L.ADG_SCEN_STEADY)
    u = m.get_state()
    g = torch.Generator().manual_seed(seed)
    m.set_state((u * (1.0 + 1e-4 * torch.rand(u.shape, generator=g, dtype=torch.float64).cuda())).contiguous())
    return m


@pytest.mark.parametrize("kind", ["walls", "periodic"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 1), (3, 1), (2, 3), (5, 3)])
def test_pairs_equal_single_nodes_bitwise(kind, nx, ny):
    from paper_1905_05524_gb300.solver import Batch
    a, b = _mesh(kind, nx, ny, 3), _mesh(kind, nx, ny, 3)
    dt = a.stable_dt(0.3)
    batch = Batch([b])
    batch.set_candidate(1)
    a.step(dt, 2)
    batch.step([dt], 2)
    assert torch.equal(a.get_state(), b.get_state())
    batch.set_candidate(3)
    a.step(dt, 2)
    batch.step([dt], 2)
    assert torch.equal(a.get_state(), b.get_state())
    batch.close()
