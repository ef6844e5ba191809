"""FP32 3D subdomains that are long in z: fewer teams to a CTA, down to one.
Created and run against the oracle, one level per pass in every mode and, where
their halos fit, in blocked passes."""
import numpy as np
import pytest

import oracle
from gpu_util import TOL, rel_linf
from test_gpu_3d import gpu_run3d
from test_gpu_3d_groups import box, modes

pytestmark = pytest.mark.gpu

# (m0, m1, m2): 8 teams fit up to 219, 4 up to 214 and 2 up to 171 planes of the
# first three shapes
COLUMNS = [(8, 8, 256), (16, 16, 256), (32, 8, 200), (16, 8, 160), (64, 4, 110), (128, 4, 110), (32, 16, 320),
           (8, 8, 900), (16, 16, 870)]
BLOCKED = [(8, 8, 256), (16, 16, 256), (16, 8, 160)]


@pytest.mark.parametrize("sub", COLUMNS)
def test_long_columns_match_oracle(sub):
    import paper_1911_05769_gb300 as at
    n = (2 * sub[0], 3 * sub[1], sub[2])
    u0 = box(n, 3)[0]
    length = tuple(0.3 * k for k in n)
    kw = dict(L=2, nu=0.2, dt=0.04)
    o = dict(P=(2, 3, 1), n_steps=9, dx=tuple(length[a] / n[a] for a in range(3)), **kw)
    passes = [(m, name, 1) for m, name in modes(at)] + ([(at.AT_FREE, "free", 2)] if sub in BLOCKED else [])
    for mode, name, spp in passes:
        g = gpu_run3d(u0, sub=sub, steps=9, dtype="f32", mode=mode, seed=7, record=True, calls=[4, 5], length=length,
                      steps_per_pass=spp, **kw)
        ref, hist = oracle.run3d(u0, delay_mode=oracle.REPLAY, replay=g["rec"], **o) if name == "free" else \
            oracle.run3d(u0, delay_mode=oracle.SEEDED if name == "seeded" else oracle.SYNC, seed=7, **o)
        assert rel_linf(g["u"], ref) <= TOL["f32"], (name, spp)
        assert np.array_equal(g["hist"], hist), (name, spp)


def test_cta_count_of_the_caller():
    """304 CTAs of 32 x 8 x 171 points: two to an SM with one team, not with two."""
    import paper_1911_05769_gb300 as at
    s = at.Solver3D((384, 96, 513), (32, 8, 171), 2, 0.1, 1e-7, max_ctas=304)
    assert s.info().ctas == 304
    s.close()


@pytest.mark.parametrize("nf", [3, 4, 5])
def test_two_ctas_of_the_system_to_an_sm(nf):
    """Planes of 1024 points, more CTAs than SMs."""
    import paper_1911_05769_gb300 as at
    from test_gpu_system3d import gpu_system
    n, sub = (256, 64, 120), (128, 8, 3)
    q0 = box(n, 5, nf)
    dx = tuple(2 * np.pi / k for k in n)
    kappa = [0.05, 0.05, 0.05, 0.02, 0.08][:nf]
    dt = 0.2 / (2 * 0.08 * sum(1 / d ** 2 for d in dx))
    kw = dict(L=2, kappa=kappa, dt=dt)
    s = at.System3D(n, sub, 2, kappa, dt)
    sms = s.info().sm_count
    s.close()
    g = gpu_system(q0, sub=sub, steps=6, dtype="f32", mode=at.AT_SEEDED, seed=7, max_ctas=2 * sms, **kw)
    ref, _ = oracle.run3d_system(q0, delay_mode=oracle.SEEDED, seed=7, P=(2, 8, 40), n_steps=6, dx=dx, **kw)
    assert rel_linf(g["q"], ref) <= TOL["f32"]
