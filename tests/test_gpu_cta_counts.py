"""CTA counts of the caller's that cannot all be resident: as many as can, where
every subdomain has a warp then, or the same with fewer tile buffers; else
refused."""
import numpy as np
import pytest

import at_workloads as W
from gpu_util import TOL, gpu_run, oracle_run, rel_linf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,M,dtype,max_ctas,stages", [(600, 1024, "f64", 1000, 0), (600, 1024, "f64", 100000, 4),
                                                       (300, 400, "f64", 300, 8), (1024, 64, "f32", 1000, 0),
                                                       (5000, 960, "f64", 304, 0), (5000, 1000, "f64", 304, 3)])
def test_counts_beyond_the_resident_ones(P, M, dtype, max_ctas, stages):
    import paper_1911_05769_gb300 as at
    N, steps = P * M, 6
    u0 = W.u0_fourier(N, modes=8, seed=1).astype(np.float32).astype(np.float64)
    _, dx = W.grid(N)
    kw = dict(P=P, order=4, L=2, nu=0.02, dt=0.2 * W.dt_rule(u0, dx, 0.02), steps=steps, forcing=0.1)
    ref, hist = oracle_run(u0, mode="seeded", seed=5, **kw)
    g = gpu_run(u0, mode=at.AT_SEEDED, seed=5, dtype=dtype, max_ctas=max_ctas, stages=stages, **kw)
    assert g["info"].ctas <= max_ctas and (g["info"].ctas == max_ctas or 4 * g["info"].ctas >= P)
    assert rel_linf(g["u"], ref) <= TOL[dtype]
    assert np.array_equal(g["hist"], hist)


def test_counts_that_stay_refused():
    import paper_1911_05769_gb300 as at
    for P, M, dtype in ((5000, 64, "f32"), (5000, 1024, "f64")):
        with pytest.raises(at.AtError) as e:
            at.Solver(P * M, P, 4, 2, 0.02, 1e-13, dtype=dtype, max_ctas=100000)
        assert e.value.code == at.AT_ERR_RESIDENCY
