"""The FP32 3D stepper with 4-point groups at the shapes where it can go wrong:
every team size (planes of 8 to 1024 points), rows of one group, planes that do
not fill their team, subdomains of 3, 4 and 5 planes (first and last plane next
to each other), faces whose word count is no multiple of 4, one and several
subdomains per team, teams without one.  Against the 3D oracles, at the FP32 bar
of the other 3D tests."""
import numpy as np
import pytest

import oracle
from gpu_util import TOL, rel_linf
from test_gpu_3d import gpu_run3d
from test_gpu_system3d import gpu_system

pytestmark = pytest.mark.gpu

# (n0, n1, n2), (m0, m1, m2), CTAs
SHAPES = [
    ((8, 4, 6), (4, 2, 3), 0),           # one group per row, 6 words an x face
    ((16, 9, 12), (8, 3, 4), 0),         # 6 groups of a 32-thread team
    ((32, 12, 10), (16, 6, 5), 1),       # 24 groups, several subdomains per team
    ((32, 32, 20), (16, 16, 5), 2),      # teams of 64
    ((64, 20, 12), (32, 10, 4), 0),      # 80 groups of a 128-thread team
    ((64, 32, 9), (32, 16, 3), 3),       # full 128-thread teams
    ((64, 64, 12), (32, 32, 4), 0),      # planes of 1024 points
    ((128, 16, 10), (128, 8, 5), 0),     # a row per warp
]


def box(n, seed, nf=1):
    rng = np.random.default_rng(seed)
    n0, n1, n2 = n
    z, y, x = np.meshgrid(*(2 * np.pi * np.arange(k) / k for k in (n2, n1, n0)), indexing="ij")
    q = np.zeros((nf, n2, n1, n0))
    for f in range(nf):
        for _ in range(4):
            a, b, c = rng.integers(1, 3, size=3)
            q[f] += rng.uniform(0.1, 0.2) * np.sin(a * x + rng.uniform(0, 6)) * np.sin(b * y + rng.uniform(0, 6)) \
                * np.sin(c * z + rng.uniform(0, 6))
    return q.astype(np.float32).astype(np.float64)


def modes(at):
    return [(at.AT_SEEDED, "seeded"), (at.AT_FREE, "free"), (at.AT_SYNC, "sync")]


@pytest.mark.parametrize("n,sub,ctas", SHAPES)
@pytest.mark.parametrize("equal", [True, False])
def test_scalar_groups_match_oracle(n, sub, ctas, equal):
    import paper_1911_05769_gb300 as at
    u0 = box(n, 3)[0]
    length = tuple(0.3 * k for k in n) if equal else tuple(0.3 * k * (1 + 0.2 * i) for i, k in enumerate(n))
    dx = tuple(length[a] / n[a] for a in range(3))
    P = tuple(n[a] // sub[a] for a in range(3))
    kw = dict(L=2, nu=0.2, dt=0.04)
    for mode, name in modes(at):
        g = gpu_run3d(u0, sub=sub, steps=15, dtype="f32", mode=mode, seed=7, max_ctas=ctas, record=True,
                      calls=[6, 9], length=length, **kw)
        o = dict(P=P, n_steps=15, dx=dx, **kw)
        ref, hist = oracle.run3d(u0, delay_mode=oracle.REPLAY, replay=g["rec"], **o) if name == "free" else \
            oracle.run3d(u0, delay_mode=oracle.SEEDED if name == "seeded" else oracle.SYNC, seed=7, **o)
        assert rel_linf(g["u"], ref) <= TOL["f32"], name
        assert np.array_equal(g["hist"], hist), name


@pytest.mark.parametrize("n,sub,ctas", SHAPES)
@pytest.mark.parametrize("nf", [3, 4, 5])
def test_system_groups_match_oracle(n, sub, ctas, nf):
    import paper_1911_05769_gb300 as at
    q0 = box(n, 5, nf)
    dx = tuple(2 * np.pi / n[a] for a in range(3))
    kappa = [0.05, 0.05, 0.05, 0.02, 0.08][:nf]
    P = tuple(n[a] // sub[a] for a in range(3))
    dt = 0.2 / (2 * 0.08 * sum(1 / d ** 2 for d in dx))
    for mode, name in modes(at):
        g = gpu_system(q0, sub=sub, L=2, kappa=kappa, dt=dt, steps=12, dtype="f32", mode=mode, seed=7, max_ctas=ctas,
                       record=True)
        o = dict(kappa=kappa, P=P, L=2, dt=dt, n_steps=12, dx=dx)
        ref, hist = oracle.run3d_system(q0, delay_mode=oracle.REPLAY, replay=g["rec"], **o) if name == "free" else \
            oracle.run3d_system(q0, delay_mode=oracle.SEEDED if name == "seeded" else oracle.SYNC, seed=7, **o)
        assert rel_linf(g["q"], ref) <= TOL["f32"], name
        assert np.array_equal(g["hist"], hist), name
