"""Fewer subdomains than processing elements: the failure knob finds the element of
the first one (in 3D: the first CTA has a subdomain like every other), so that
its neighbours' bounded waits run out, and runs agree with the oracle."""
import numpy as np
import pytest
import torch

import at_workloads as W
import oracle
from gpu_util import TOL, gpu_run, oracle_run, rel_linf
from test_gpu_3d import gpu_run3d
from test_gpu_3d_groups import box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,M,dtype", [(2, 64, "f64"), (16, 256, "f64"), (150, 64, "f32"), (600, 64, "f64")])
@pytest.mark.parametrize("spp", [1, 3])
def test_first_element_is_found(P, M, dtype, spp):
    import paper_1911_05769_gb300 as at
    u0 = W.u0_two_modes(P * M)
    _, dx = W.grid(P * M)
    kw = dict(P=P, order=2, L=2, nu=0.02, dt=0.1 * W.dt_rule(u0, dx, 0.02), steps=60, dtype=dtype, mode=at.AT_FREE,
              steps_per_pass=spp)
    g = gpu_run(u0, flags=at.AT_FLAG_TEST_SKIP_PUBLISH, test_skip_step=5, timeout_ns=20_000_000, check=False, **kw)
    assert g["rc"] == at.AT_ERR_TIMEOUT
    g = gpu_run(u0, record=True, **kw)
    kw = {k: v for k, v in kw.items() if k not in ("dtype", "mode", "steps_per_pass")}
    u0 = u0.astype(np.float32 if dtype == "f32" else np.float64)
    ref, hist = oracle_run(u0, mode="replay", delays=g["rec"], **kw)
    assert rel_linf(g["u"], ref) <= TOL[dtype]
    assert np.array_equal(g["hist"], hist)


@pytest.mark.parametrize("sub", [(8, 8, 8), (16, 16, 16), (32, 16, 8)])
def test_first_cta_takes_part_3d(sub):
    """FP32 planes of 64, 256 and 512 points: CTAs of 8, 4 and 2 teams."""
    import paper_1911_05769_gb300 as at
    n = tuple(3 * m for m in sub)
    u0 = box(n, 3)[0]
    length = tuple(0.3 * k for k in n)
    kw = dict(sub=sub, L=2, nu=0.2, dt=0.04, dtype="f32", mode=at.AT_FREE, length=length)
    s = at.Solver3D(n, sub, 2, 0.2, 0.04, length=length, flags=at.AT_FLAG_TEST_SKIP_PUBLISH, test_skip_step=4,
                    timeout_ns=20_000_000)
    s.set_state(torch.from_numpy(np.ascontiguousarray(u0)).ravel())
    s.step(40, at.AT_FREE)
    assert s.status() == at.AT_ERR_TIMEOUT
    s.close()
    g = gpu_run3d(u0, steps=15, record=True, **kw)
    ref, hist = oracle.run3d(u0, delay_mode=oracle.REPLAY, replay=g["rec"], P=(3, 3, 3), n_steps=15, L=2, nu=0.2,
                             dt=0.04, dx=tuple(length[a] / n[a] for a in range(3)))
    assert rel_linf(g["u"], ref) <= TOL["f32"]
    assert np.array_equal(g["hist"], hist)
