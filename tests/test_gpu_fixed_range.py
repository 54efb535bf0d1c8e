"""The FP64 step far from 1: multiplying rho, rho v, rho E and mu by a power of
two scales every term of the equations, and every operation of the step is
exact under that scaling, down to states of 2^-850 (components of 2^-900) and
up to 2^850."""
import pytest
import torch

from tests.test_fixed_point import _flow, _steady

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degree", [1, 3, 5, 7])
@pytest.mark.parametrize("power", [-850, 850])
def test_step_scales_bitwise(degree, power):
    out = []
    for s in (1.0, 2.0 ** power):
        cfg, m = _steady(degree, 3, 2, s, False)
        m.set_state((_flow(cfg, degree) * s).cuda())
        for _ in range(2):
            m.step(1e-3)
        out.append(m.get_state().cpu())
        m.close()
    assert torch.isfinite(out[0]).all()
    assert torch.equal(out[0] * 2.0 ** power, out[1])
