"""Bounded waits of the steppers that run out: the first CTA stops publishing
(test knob), every kernel form returns with AT_ERR_TIMEOUT latched, and the
next run on the context is right."""
import numpy as np
import pytest
import torch

import at_workloads as W
import oracle
from gpu_util import TOL, gpu_run, oracle_run, rel_linf
from test_gpu_3d_groups import box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sub,dtype", [((8, 8, 4), "f32"), ((16, 16, 4), "f32"), ((32, 16, 4), "f32"),
                                       ((32, 32, 4), "f32"), ((12, 8, 4), "f32"), ((16, 8, 4), "f64")])
@pytest.mark.parametrize("mode_name", ["seeded", "free"])
@pytest.mark.parametrize("skip", [0, 5])
def test_3d_teams_leave_together(sub, dtype, mode_name, skip):
    """Planes of 64 to 1024 points (CTAs of 8, 4, 2 and 1 teams, and the kernel
    of single columns); the knob acts from the first level on, so that the
    first tiles' waits run out, or after some."""
    import paper_1911_05769_gb300 as at
    mode = at.AT_SEEDED if mode_name == "seeded" else at.AT_FREE
    n = (4 * sub[0], 4 * sub[1], 6 * sub[2])
    u0 = box(n, 9)[0]
    length = tuple(0.3 * k for k in n)
    for flags in (at.AT_FLAG_TEST_SKIP_PUBLISH, 0):
        s = at.Solver3D(n, sub, 2, 0.2, 0.04, dtype=dtype, length=length, seed=3, max_ctas=3, flags=flags,
                        test_skip_step=skip, timeout_ns=20_000_000 if flags else 0)
        s.set_state(torch.from_numpy(np.ascontiguousarray(u0)).ravel())
        s.step(15, mode if flags else at.AT_SEEDED)
        if flags:
            assert s.status() == at.AT_ERR_TIMEOUT
            assert "timed out" in at.at_last_error()
        else:
            out = s.state().double().cpu().numpy().reshape(u0.shape)
        s.close()
    ref, _ = oracle.run3d(u0, delay_mode=oracle.SEEDED, seed=3, P=(4, 4, 6), n_steps=15, L=2, nu=0.2, dt=0.04,
                          dx=tuple(length[a] / n[a] for a in range(3)))
    assert rel_linf(out, ref) <= TOL[dtype]


@pytest.mark.parametrize("P", [2, 5, 16, 17, 200])
@pytest.mark.parametrize("M,order,dtype", [(32, 2, "f64"), (64, 4, "f64"), (100, 4, "f32"), (256, 2, "f64"), (1024, 4, "f32")])
@pytest.mark.parametrize("skip", [0, 7])
def test_one_subdomain_per_cta_leaves_together(P, M, order, dtype, skip):
    """Prescribed delays with a CTA per subdomain, of one to eight warps, through
    a cluster (P <= 16) and through the ring."""
    import paper_1911_05769_gb300 as at
    u0 = W.u0_two_modes(P * M)
    u0 = u0.astype(np.float32 if dtype == "f32" else np.float64).astype(np.float64)
    _, dx = W.grid(P * M)
    kw = dict(P=P, order=order, L=2, nu=0.02, dt=0.1 * W.dt_rule(u0, dx, 0.02), steps=80, seed=3)
    g = gpu_run(u0, mode=at.AT_SEEDED, dtype=dtype, flags=at.AT_FLAG_TEST_SKIP_PUBLISH, test_skip_step=skip,
                timeout_ns=20_000_000, check=False, **kw)
    assert g["rc"] == at.AT_ERR_TIMEOUT
    # levels up to the one published run
    g = gpu_run(u0, mode=at.AT_SEEDED, dtype=dtype, flags=at.AT_FLAG_TEST_SKIP_PUBLISH, test_skip_step=80, **kw)
    ref, hist = oracle_run(u0, mode="seeded", **kw)
    assert rel_linf(g["u"], ref) <= TOL[dtype]
    assert np.array_equal(g["hist"], hist)


@pytest.mark.parametrize("P,M,order,dtype", [(2, 64, 2, "f64"), (5, 100, 4, "f64"), (16, 1024, 2, "f32"), (300, 64, 4, "f32")])
@pytest.mark.parametrize("back", [0, 1, 9])
def test_adjoint_messages_time_out(P, M, order, dtype, back):
    """Subdomain 0 leaves out the intervals of 10 levels that start `back` or
    more backward steps in: its neighbours' waits for its messages run out;
    without the knob the gradient is the oracle's."""
    from paper_1911_05769_gb300 import AT_ERR_TIMEOUT, AT_FLAG_TEST_SKIP_PUBLISH, AT_OK, AT_SEEDED, Solver, binding as B
    from test_gpu_adjoint import oracle_adjoint, problem
    pr = problem(N=P * M, P=P, order=order, L=2, steps=24, nu=0.02 if P * M > 400 else 0.2)
    pr["dt"] *= 0.5
    if dtype == "f32":
        for k in ("u0", "lam_T"):
            pr[k] = pr[k].astype(np.float32).astype(np.float64)
    tdt = torch.float64 if dtype == "f64" else torch.float32
    n, interval = pr["steps"], 10
    for flags in (AT_FLAG_TEST_SKIP_PUBLISH, 0):
        s = Solver(pr["N"], P, order, 2, pr["nu"], pr["dt"], dtype=dtype, seed=pr["seed"], flags=flags,
                   test_skip_step=n + back, timeout_ns=20_000_000 if flags else 0)
        s.set_state(pr["u0"])
        ckpt = torch.empty(B.at_checkpoint_bytes(s.h, n, interval), dtype=torch.uint8, device="cuda")
        assert B.at_step_checkpointed(s.h, n, AT_SEEDED, None, interval, ckpt.data_ptr()) == AT_OK
        assert s.status() == AT_OK
        lam = torch.from_numpy(pr["lam_T"]).to(tdt).cuda()
        nb = B.at_adjoint_workspace_bytes(s.h, interval)
        ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
        rc, _ = B.at_adjoint(s.h, n, AT_SEEDED, None, interval, ckpt.data_ptr(), ws.data_ptr(), nb, lam.data_ptr())
        assert rc == (AT_ERR_TIMEOUT if flags else AT_OK)
        s.close()
    _, olam0, _ = oracle_adjoint(pr, mode=oracle.SEEDED)
    assert rel_linf(lam.double().cpu().numpy(), olam0) <= TOL[dtype]
