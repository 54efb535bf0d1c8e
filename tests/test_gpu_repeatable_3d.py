"""The 3D step gives the same bits every time: its corrector is scheduled while
the predictor finishes and must read none of its outputs before the wait."""
import pytest
import torch

from paper_1905_05524_gb300 import _lib as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [L.ADG_PREC_MIXED, L.ADG_PREC_FP64])
@pytest.mark.parametrize("degree", [1, 2, 3, 4])
def test_runs_are_bitwise_equal(degree, precision):
    from paper_1905_05524_gb300.solver import Mesh3, bubble3d_config
    cfg = bubble3d_config(degree=degree, n=3, mu=0.5)
    cfg.ny, cfg.nz, cfg.precision = 4, 5, precision
    first = None
    for _ in range(8):
        m = Mesh3(cfg)
        m.init_scenario(L.ADG_SCEN_COSINE)
        m.step(m.stable_dt(0.25), 16)
        u = m.get_state()
        m.close()
        assert first is None or torch.equal(u, first)
        first = u
