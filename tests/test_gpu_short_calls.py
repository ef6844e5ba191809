"""Forced runs with a few hundred subdomains: short and long calls take different
kernels (and calls of one solver take turns between them), with the oracle's
result and the same bits whatever the calls' lengths; and no more FP64 CTAs than
the subdomains need, so that the start of a call stays short."""
import numpy as np
import pytest

import at_workloads as W
from gpu_util import TOL, gpu_run, oracle_run, rel_linf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,M,dtype", [(170, 64, "f32"), (300, 256, "f32"), (600, 1024, "f32"), (1000, 64, "f64"),
                                       (600, 256, "f64"), (470, 100, "f64")])
@pytest.mark.parametrize("order", [2, 4])
def test_call_lengths_give_the_same_bits(P, M, dtype, order):
    import paper_1911_05769_gb300 as at
    u0 = W.u0_fourier(P * M, modes=8, seed=2).astype(np.float32).astype(np.float64)
    _, dx = W.grid(P * M)
    kw = dict(P=P, order=order, L=3, nu=0.02, dt=0.2 * W.dt_rule(u0, dx, 0.02), steps=170, forcing=0.1)
    ref, hist = oracle_run(u0, mode="seeded", seed=5, **kw)
    one = None
    for calls in ([170], [1, 3, 150, 2, 14], [1] * 20 + [150]):
        g = gpu_run(u0, mode=at.AT_SEEDED, seed=5, dtype=dtype, calls=calls, **kw)
        assert rel_linf(g["u"], ref) <= TOL[dtype]
        assert np.array_equal(g["hist"], hist)
        assert one is None or np.array_equal(one, g["u"])
        one = g["u"]


@pytest.mark.parametrize("P,M", [(16, 256), (300, 1024), (600, 1000), (600, 1024)])
def test_no_more_ctas_than_subdomains_need(P, M):
    import paper_1911_05769_gb300 as at
    s = at.Solver(P * M, P, 4, 2, 0.02, 1e-13, dtype="f64", forcing_amp=0.1)
    i = s.info()
    assert i.ctas == min(P, -(-P // (4 * i.sm_count)) * i.sm_count)
    s.close()
