"""Tiles of the 1D stepper at the sizes where its lane layout can go wrong:
lanes of whole groups that fill the warp or leave lanes empty, runs that end
inside a lane, tiles within one lane, every run length and swizzle; elements of
one subdomain (kept in registers), of two and of several; delay bounds beyond
the 16 ring entries read at once.  Every run against the oracle with the run's
own delays, at the bars of the other GPU tests."""
import numpy as np
import pytest

import at_workloads as W
from gpu_util import TOL, gpu_run, oracle_run, rel_linf

pytestmark = pytest.mark.gpu

# points per subdomain: one lane (4), partly filled warps (64, 100, 400), full
# warps (128, 256, 512, 1024), runs of 2..8 groups with a short last one
SIZES = [4, 12, 64, 100, 128, 132, 200, 256, 260, 380, 400, 500, 512, 768, 1000, 1020, 1024]


@pytest.mark.parametrize("M", SIZES)
@pytest.mark.parametrize("order,dtype,forcing", [(2, "f64", 0.0), (4, "f64", 0.1), (2, "f32", 0.1), (4, "f32", 0.1)])
def test_tile_sizes_match_oracle(require_gpu, M, order, dtype, forcing):
    import paper_1911_05769_gb300 as at
    P, L, steps = 11, 3, 26
    N = P * M
    u0 = W.u0_fourier(N, modes=8, seed=M)
    if dtype == "f32":
        u0 = u0.astype(np.float32).astype(np.float64)
    _, dx = W.grid(N)
    nu = 0.02 if N > 500 else 0.2
    dt = 0.5 * W.dt_rule(u0, dx, nu)
    kw = dict(P=P, order=order, L=L, nu=nu, dt=dt, steps=steps, forcing=forcing)
    # (1 CTA: 2-3 subdomains per element; 0: one each, kept in registers)
    for mode, spp, ctas, calls in (("seeded", 1, 1, [9, 17]), ("seeded", 1, 0, None), ("free", L + 1, 1, [3, 23]),
                                   ("free", L + 1, 0, None), ("free", 1, 2, None), ("sync", 1, 0, None),
                                   ("sync", 2 if M < 12 else L + 1, 1, None)):
        m = {"seeded": at.AT_SEEDED, "free": at.AT_FREE, "sync": at.AT_SYNC}[mode]
        g = gpu_run(u0, mode=m, seed=5, dtype=dtype, max_ctas=ctas, steps_per_pass=spp, record=True, calls=calls, **kw)
        if mode == "free":
            ref, hist = oracle_run(u0, mode="replay", delays=g["rec"], **kw)
        else:
            ref, hist = oracle_run(u0, mode=mode, seed=5, **kw)
        assert rel_linf(g["u"], ref) <= TOL[dtype], (mode, spp, ctas)
        assert np.array_equal(g["hist"], hist), (mode, spp, ctas)


@pytest.mark.parametrize("M", [4, 100, 400, 500, 1024])
@pytest.mark.parametrize("order", [2, 4])
def test_compensated_tiles_match_oracle(require_gpu, M, order):
    import paper_1911_05769_gb300 as at
    P, L, steps = 7, 2, 20
    N = P * M
    u0 = W.u0_fourier(N, modes=8, seed=M).astype(np.float32).astype(np.float64)
    _, dx = W.grid(N)
    nu = 0.02 if N > 500 else 0.2
    kw = dict(P=P, order=order, L=L, nu=nu, dt=0.5 * W.dt_rule(u0, dx, nu), steps=steps, forcing=0.1)
    for mode, spp, ctas in ((at.AT_SEEDED, 1, 1), (at.AT_FREE, L + 1, 0)):
        g = gpu_run(u0, mode=mode, seed=3, dtype="f32", flags=at.AT_FLAG_COMPENSATED, max_ctas=ctas,
                    steps_per_pass=spp, record=True, **kw)
        ref, _ = oracle_run(u0, mode="replay", delays=g["rec"], **kw)
        # (hi alone: one rounding to FP32, 2^-24 of the largest value)
        assert rel_linf(g["u"], ref) <= 2.0 ** -23
        assert rel_linf(g["u"] + g["lo"], ref) <= TOL["f32"] * 0.01


@pytest.mark.parametrize("L", [13, 14, 16])
def test_free_running_delay_bounds_beyond_one_read(require_gpu, L):
    import paper_1911_05769_gb300 as at
    P, M, steps = 24, 64, 60
    u0 = W.u0_fourier(P * M, modes=8, seed=L)
    _, dx = W.grid(P * M)
    kw = dict(P=P, order=2, L=L, nu=0.02, dt=0.1 * W.dt_rule(u0, dx, 0.02), steps=steps)
    for spp in (1, 5, L + 1):
        g = gpu_run(u0, mode=at.AT_FREE, dtype="f64", max_ctas=2, steps_per_pass=spp, record=True, **kw)
        assert g["rec"].min() >= 0 and g["rec"].max() <= L
        ref, hist = oracle_run(u0, mode="replay", delays=g["rec"], **kw)
        assert rel_linf(g["u"], ref) <= TOL["f64"]
        assert np.array_equal(g["hist"], hist)


@pytest.mark.parametrize("stages", [2, 3, 4])
@pytest.mark.parametrize("per_pe", [2, 3, 5, 15, 16, 17, 35])
def test_one_level_passes_turn(require_gpu, per_pe, stages):
    """Passes of one level alternate their direction too: the delays drawn 16
    tiles at a time follow the turns (blocks that end at, before and after a
    turn, and that hold several), the grid barrier of the synchronous mode
    stands before a turn tile, and every call starts forward again."""
    import paper_1911_05769_gb300 as at
    P, M, L = 8 * per_pe, 64, 3
    u0, dt = _turn_setup(P * M)
    kw = dict(P=P, order=4, L=L, nu=0.02, dt=dt, steps=31, forcing=0.1)
    for mode, name in ((at.AT_SEEDED, "seeded"), (at.AT_SYNC, "sync")):
        g = gpu_run(u0, mode=mode, seed=11, max_ctas=2, stages=stages, record=True, calls=[1, 17, 13],
                    steps_per_pass=1, **kw)
        ref, hist = oracle_run(u0, mode=name, seed=11, **kw)
        assert g["info"].ctas == 2
        assert rel_linf(g["u"], ref) <= TOL["f64"], name
        assert np.array_equal(g["hist"], hist), name


def _turn_setup(N):
    u0 = W.u0_fourier(N, modes=8, seed=N)
    _, dx = W.grid(N)
    return u0, 0.5 * W.dt_rule(u0, dx, 0.02)
