"""dJ/dnu of the adjoint against the oracle's: partly filled warps, one-lane tiles,
short last runs, lanes beyond a full tile, sums over intervals, and the blocks
that walk the subdomains where not every one has a warp."""
import numpy as np
import pytest

import oracle
from gpu_util import TOL
from test_gpu_adjoint import gpu_adjoint, oracle_adjoint, problem

pytestmark = pytest.mark.gpu


def bound(pr, dtype):
    """The bar of the other tests on the size of the sum of the terms' absolute
    values (steps x points, the adjoint and the second differences as they are at
    the ends they are known at), and the rounding of the levels themselves, half an
    ulp in every value of every second difference."""
    u, dx = pr["u0"], 2 * np.pi / pr["N"]
    if pr["order"] == 2:
        b, q, beta = np.roll(u, 1) + np.roll(u, -1) - 2 * u, 1, 4
    else:
        b, q = 16 * (np.roll(u, 1) + np.roll(u, -1)) - (np.roll(u, 2) + np.roll(u, -2)) - 30 * u, 12
        beta = 64
    rounding = beta * (2.0 ** -24 if dtype == "f32" else 2.0 ** -53) * np.max(np.abs(u))
    return pr["steps"] * np.sum(np.abs(pr["lam_T"])) * (TOL[dtype] * np.max(np.abs(b)) + rounding) * pr["dt"] / (q * dx * dx)


@pytest.mark.parametrize("order,M,P", [(2, 4, 7), (4, 4, 7), (2, 100, 5), (4, 256, 1), (4, 400, 2), (2, 500, 9),
                                       (4, 768, 3), (2, 1024, 4), (4, 1020, 3), (4, 960, 5)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_viscosity_gradient(order, M, P, dtype):
    from paper_1911_05769_gb300 import AT_SEEDED
    pr = problem(N=P * M, P=P, order=order, L=3, steps=23, nu=0.02 if P * M > 400 else 0.2, seed=M)
    pr["dt"] *= 0.5
    if dtype == "f32":
        for k in ("u0", "lam_T"):
            pr[k] = pr[k].astype(np.float32).astype(np.float64)
    _, _, odnu = oracle_adjoint(pr, mode=oracle.SEEDED)
    for interval in (1, 3, 11, 40):
        _, _, dnu, _ = gpu_adjoint(pr, mode=AT_SEEDED, interval=interval, dtype=dtype)
        assert abs(dnu - odnu) <= bound(pr, dtype), (interval, dnu, odnu)


def test_viscosity_gradient_of_more_subdomains_than_warps():
    from paper_1911_05769_gb300 import AT_SEEDED
    pr = problem(N=4 * 20000, P=20000, order=2, L=2, steps=12, nu=0.02)
    _, _, odnu = oracle_adjoint(pr, mode=oracle.SEEDED)
    _, _, dnu, _ = gpu_adjoint(pr, mode=AT_SEEDED, interval=5)
    assert abs(dnu - odnu) <= bound(pr, "f64"), (dnu, odnu)
