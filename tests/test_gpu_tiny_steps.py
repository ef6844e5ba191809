"""FP32 runs whose time step is so short that the stencil's factors are 0 in FP32:
the state stays what it was."""
import numpy as np
import pytest

import at_workloads as W
from gpu_util import gpu_ensemble_run, gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("forcing", [0.0, 0.1])
@pytest.mark.parametrize("flags", [0, 32])
def test_factors_below_fp32(order, forcing, flags):
    import paper_1911_05769_gb300 as at
    P, M = 5, 100
    u0 = W.u0_two_modes(P * M).astype(np.float32)
    for mode, ctas in ((at.AT_SEEDED, 0), (at.AT_SEEDED, 2), (at.AT_FREE, 0)):
        g = gpu_run(u0, P=P, order=order, L=2, nu=0.02, dt=1e-60, steps=9, dtype="f32", mode=mode, max_ctas=ctas,
                    forcing=forcing, flags=flags)
        assert np.array_equal(g["u"], u0)


@pytest.mark.parametrize("flags", [0, 32])
def test_factors_below_fp32_ensemble(flags):
    import paper_1911_05769_gb300 as at
    inst = [dict(n=512, L=1, nu=0.01, dt=1e-60, bc=at.AT_BC_PERIODIC, length=2 * np.pi, origin=0.0, tanh_a=0.5,
                 tanh_c=0.1, tanh_xc=0.0, seed=j) for j in range(3)]
    u0 = W.ensemble_field(inst).astype(np.float32)
    g = gpu_ensemble_run(inst, M=128, order=2, steps=9, dtype="f32", mode=at.AT_FREE, steps_per_pass=2, flags=flags)
    assert np.array_equal(g["u"], u0)
