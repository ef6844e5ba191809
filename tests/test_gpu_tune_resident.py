"""at_tune with prescribed delays where every subdomain has a CTA of its own: that
kernel is timed once, against every shape of the general one, and the choice does
not touch the results or the other modes' shapes."""
import numpy as np
import pytest

import at_workloads as W
import oracle
from gpu_util import TOL, rel_linf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,M,forcing", [(16, 256, 0.0), (16, 64, 0.1), (1000, 256, 0.0)])
def test_tuning_with_prescribed_delays(P, M, forcing):
    from paper_1911_05769_gb300 import AT_SEEDED, Solver
    u0 = W.u0_two_modes(P * M)
    _, dx = W.grid(P * M)
    dt = 0.2 * W.dt_rule(u0, dx, 0.02)
    s = Solver(P * M, P, 2, 2, 0.02, dt, dtype="f64", seed=7, forcing_amp=forcing)
    before = s.info()
    s.set_state(u0)
    tried = 0
    for _ in range(2):
        t = s.tune(10, AT_SEEDED)
        tried += t.n_tried
        if P == 16:
            # one CTA count, 2 to 4 tile buffers, and the kernel without them
            assert t.n_tried == 4
        assert t.best_ms <= t.first_ms
        after = s.info()
        assert (after.ctas, after.stages) == (t.ctas, t.stages)
    s.step(25, AT_SEEDED)
    total = s.info().step
    assert total == 25 + 3 * 10 * tried
    ref, hist = oracle.run(u0, P=P, order=2, L=2, nu=0.02, dt=dt, n_steps=total, delay_mode=oracle.SEEDED, seed=7,
                           forcing_amp=forcing)
    assert rel_linf(s.state().cpu().numpy(), ref) <= TOL["f64"]
    assert np.array_equal(s.delay_stats()[0], hist)
    assert before.ctas <= P
    s.close()
