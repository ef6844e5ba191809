"""Runs with prescribed delays of up to 16 subdomains hand their boundary values
over inside one thread block cluster: the same values to the last bit, delay
counts and ring levels as the general stepper (which a CTA count of the caller
selects), over calls that mix modes, short calls and every delay bound."""
import pytest
import torch

import at_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("order,forcing", [(2, 0.0), (2, 0.1), (4, 0.0), (4, 0.1)])
@pytest.mark.parametrize("P,M,L", [(2, 64, 0), (2, 1024, 3), (3, 100, 16), (5, 1020, 3), (8, 512, 2), (16, 128, 3),
                                   (16, 1024, 1), (17, 64, 2)])
def test_cluster_equals_general_stepper(dtype, order, forcing, P, M, L):
    from paper_1911_05769_gb300 import AT_SEEDED, AT_SYNC, Solver
    N = P * M
    u0 = W.u0_two_modes(N)
    _, dx = W.grid(N)
    dt = W.dt_rule(u0, dx, 0.02) / (1 + L) ** 2          # (long delays are unstable at the full step)
    out = []
    for max_ctas in (0, P):
        s = Solver(N, P, order, L, 0.02, dt, dtype=dtype, forcing_amp=forcing, seed=77, max_ctas=max_ctas)
        s.set_state(u0)
        states = []
        for steps, mode in ((1, AT_SEEDED), (2, AT_SEEDED), (70, AT_SEEDED), (3, AT_SYNC), (1, AT_SEEDED), (90, AT_SEEDED)):
            s.step(steps, mode)
            states.append(s.state().clone())
        out.append((states, s.delay_stats()))
        s.close()
    for a, b in zip(*[o[0] for o in out]):
        assert torch.isfinite(a).all() and torch.equal(a, b)
    assert list(out[0][1][0]) == list(out[1][1][0])
