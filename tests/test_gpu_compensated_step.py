"""One step of the compensated state where increments are far below its lo words:
hi + lo changes by the increment, formed apart, rounded once at lo's magnitude."""
import numpy as np
import pytest

import at_workloads as W

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("A", [0.0, 0.1])
@pytest.mark.parametrize("M", [64, 100, 512])
def test_increment_is_rounded_once(order, A, M):
    """1000 steps of dt = 1e-10 fill the lo words (up to 2^-25 for values near 1);
    one more adds the exact increment to within half an ulp of the new lo word and
    8 roundings of the increment's terms, which are a few hundredths of that."""
    from paper_1911_05769_gb300 import AT_FLAG_COMPENSATED, AT_SYNC, Solver
    P, nu, dt = 6, 0.02, 1e-10
    N = P * M
    x, dx = W.grid(N)
    u0 = (1.0 + 0.3 * np.sin(x) + 0.2 * np.sin(5 * x + 1)).astype(np.float32)
    s = Solver(N, P, order, 2, nu, dt, dtype="f32", forcing_amp=A, flags=AT_FLAG_COMPENSATED)
    s.set_state(u0)
    s.step(1000, AT_SYNC)
    state = []
    for _ in range(2):
        state.append([t.cpu().numpy().astype(np.longdouble) for t in (s.state(), s.state_error())])
        s.step(1, AT_SYNC)
    s.close()
    (h0, l0), (h1, l1) = state
    u = h0 + l0

    def at(k):
        return np.roll(u, -k)

    if order == 2:
        a, b, q = at(1) - at(-1), at(1) + at(-1) - 2 * u, (2, 1)
    else:
        a = 8 * (at(1) - at(-1)) - (at(2) - at(-2))
        b, q = 16 * (at(1) + at(-1)) - (at(2) + at(-2)) - 30 * u, (12, 12)
    adv, vis, frc = dt / (q[0] * dx) * u * a, nu * dt / (q[1] * dx * dx) * b, dt * A * np.sin(x)
    du = vis - adv + frc
    err = np.abs((h1 - h0) + (l1 - l0) - du)
    half = np.spacing(np.abs(l0 + du).astype(np.float32) * np.float32(1 + 1e-6)).astype(np.float64) / 2
    bound = half + 8 * EPS * (np.abs(vis) + np.abs(adv) + np.abs(frc))
    assert np.all(err <= bound), float(np.max(err / bound))
