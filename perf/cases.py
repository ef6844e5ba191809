"""Performance cases of the AT solver: what a user has it do, through the
package's public classes and ``at_run``.

Every pass of a stepping case is a whole run as a program makes it: set the
initial field, advance ``steps`` levels, take the state back.  The adjoint
cases run the differentiable entry point forward and backward.  Inputs are
seeded synthetic fields of the kinds the package's workloads use (Fourier
modes, travelling tanh fronts, random-phase k^-5/3 fields), made on the GPU.

``exact`` restates each run in 64-bit torch.  Prescribed (seeded) delays are
drawn and applied as the scheme defines them.  Free-running runs have many
correct results; they are listed only where the time step is so short that the
delayed halos differ from the undelayed ones by less than the state's
rounding (or, in three dimensions, by a few units of it), and ``exact`` takes
delay 0 there.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1911_05769_gb300 as at

TWO_PI = 2.0 * math.pi
MODES = {"sync": at.AT_SYNC, "seeded": at.AT_SEEDED, "free": at.AT_FREE}


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a short double-precision run, as in a unit test,
        # a convergence study or a parameter scan; launch and hand-over latency
        dict(name="run1d_n1024_f64", kind="run1d", P=16, M=64, order=4, L=3, dtype="f64", mode="seeded", spp=1,
             forced=True, comp=False, steps=120),
        # the paper-like small domain (4096 points on 16 elements, 1000
        # steps): every step waits for the neighbours
        dict(name="run1d_n4096_f64", kind="run1d", P=16, M=256, order=2, L=2, dtype="f64", mode="seeded", spp=1,
             forced=False, comp=False, steps=1000),
        # a mid-size run whose subdomains are no multiple of a warp's 128 points
        dict(name="run1d_ragged_f32_free", kind="run1d", P=5000, M=500, order=4, L=3, dtype="f32", mode="free",
             spp=4, forced=True, comp=False, steps=400),
        # the large forced run, free-running in passes of L + 1 levels: the
        # production mode of the method
        dict(name="run1d_n2p26_f32_free", kind="run1d", P=65536, M=1024, order=4, L=3, dtype="f32", mode="free",
             spp=4, forced=True, comp=False, steps=100),
        # the same equation with prescribed delays (reproducible runs), one
        # level per pass
        dict(name="run1d_n2p25_f32_seeded", kind="run1d", P=32768, M=1024, order=4, L=3, dtype="f32", mode="seeded",
             spp=1, forced=True, comp=False, steps=100),
        # double precision at size, free-running in passes
        dict(name="run1d_n2p22_f64_free", kind="run1d", P=4096, M=1024, order=4, L=3, dtype="f64", mode="free",
             spp=4, forced=True, comp=False, steps=40),
        # the compensated FP32 state, for runs of many short steps
        dict(name="run1d_n2p24_comp_free", kind="run1d", P=16384, M=1024, order=4, L=3, dtype="f32", mode="free",
             spp=4, forced=True, comp=True, steps=100),
        # 2048 independent travelling waves of uneven sizes in one launch
        dict(name="ensemble_2048_f32_free", kind="ensemble", inst=2048, M=256, lo=10, hi=16, order=2, dtype="f32",
             mode="free", spp=4, tile=4, comp=False, steps=100),
        # the gradient of a terminal loss through 200 seeded steps
        dict(name="adjoint_n2p20_f32", kind="adjoint", P=1024, M=1024, order=2, L=2, dtype="f32", steps=200,
             interval=100),
        # the 3D scalar workload, free-running in passes of L + 1 levels
        dict(name="run3d_n512_f32_free", kind="run3d", n0=512, n1=512, n2=512, m0=32, m1=32, m2=32, L=2,
             dtype="f32", mode="free", spp=3, fields=1, cfl=0.2, steps=24),
        # 3D with prescribed delays on an uneven box, one level per pass
        dict(name="run3d_box_f32_seeded", kind="run3d", n0=384, n1=256, n2=288, m0=32, m1=32, m2=32, L=2,
             dtype="f32", mode="seeded", spp=1, fields=1, cfl=0.2, steps=40),
        # velocity and two passive scalars in 3D (the full system)
        dict(name="system3d_n256_f32_free", kind="run3d", n0=256, n1=256, n2=256, m0=16, m1=16, m2=16, L=2,
             dtype="f32", mode="free", spp=1, fields=5, cfl=0.2, steps=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run1d", "run1d", "run1d", "ensemble", "adjoint", "run3d", "system3d"])
    if kind == "run1d":
        N = _log_int(rng, 1 << 10, 1 << 26)
        M = rng.choice([64, 100, 128, 200, 256, 380, 500, 512, 768, 1000, 1020, 1024, 1024])
        P = max(4, N // M)
        N = P * M
        dtype = rng.choice(["f32", "f32", "f64"])
        order, L = rng.choice([2, 4]), rng.randint(1, 3)
        # (free-running at sizes whose time step makes the delays invisible)
        mode = rng.choice(["free", "free", "seeded", "sync"] if N >= 1 << 20 else ["seeded", "seeded", "sync"])
        spp = rng.choice([1, L + 1, L + 1]) if mode != "seeded" else 1
        comp = dtype == "f32" and rng.random() < 0.2
        most = 4e9 if dtype == "f32" else 1e8
        steps = max(10, min(_log_int(rng, 30, 1000), int(most / N)))
        if N * steps > 1.5 * most:
            P = max(4, int(most / steps) // M)
        return dict(kind="run1d", P=P, M=M, order=order, L=L, dtype=dtype, mode=mode, spp=spp,
                    forced=rng.random() < 0.5, comp=comp, steps=steps)
    if kind == "ensemble":
        M = rng.choice([64, 128, 256, 256, 512])
        mode = rng.choice(["free", "sync"])
        tile = 1 if M == 64 else rng.choice([1, 2, 1024 // M if M > 256 else 4])
        return dict(kind="ensemble", inst=_log_int(rng, 64, 2048), M=M, lo=rng.randint(10, 11),
                    hi=rng.randint(13, 16), order=2, dtype="f32", mode=mode, spp=rng.choice([1, 4]) if mode == "free"
                    else 1, tile=tile, comp=rng.random() < 0.2, steps=rng.randint(20, 100))
    if kind == "adjoint":
        dtype = rng.choice(["f32", "f32", "f64"])
        M = rng.choice([256, 500, 512, 1000, 1024])
        N = _log_int(rng, 1 << 13, 1 << 20 if dtype == "f32" else 1 << 16)
        return dict(kind="adjoint", P=max(4, N // M), M=M, order=rng.choice([2, 2, 4]) if dtype == "f64" else 2, L=2,
                    dtype=dtype, steps=rng.randint(60, 200), interval=rng.choice([25, 50, 100]))
    if kind == "run3d":
        m0, m1, m2 = rng.choice([(32, 32, 32), (32, 32, 32), (32, 16, 24), (16, 16, 16), (64, 16, 20), (32, 32, 20)])
        mode = rng.choice(["free", "seeded", "sync"])
        dtype = rng.choice(["f32", "f32", "f32", "f64"])
        top = 320 if dtype == "f32" else 160
        n = [m * max(2, round(rng.uniform(256, top) / m if mode == "free" and dtype == "f32" else
                              rng.uniform(96, top) / m)) for m in (m0, m1, m2)]
        if mode == "free" and dtype == "f64":
            mode = "seeded"
        return dict(kind="run3d", n0=n[0], n1=n[1], n2=n[2], m0=m0, m1=m1, m2=m2, L=2, dtype=dtype, mode=mode,
                    spp=rng.choice([1, 3, 3]) if mode == "free" else 1, fields=1, cfl=0.05 if mode == "free" else 0.2,
                    steps=rng.randint(8, 24))
    m = rng.choice([(16, 16, 16), (16, 16, 16), (32, 16, 16), (32, 8, 12)])
    n = [a * max(2, round(rng.uniform(96, 256) / a)) for a in m]
    mode = rng.choice(["seeded", "sync"])
    return dict(kind="run3d", n0=n[0], n1=n[1], n2=n[2], m0=m[0], m1=m[1], m2=m[2], L=2,
                dtype=rng.choice(["f32", "f32", "f64"]) if n[0] * n[1] * n[2] < 1 << 22 else "f32", mode=mode, spp=1,
                fields=rng.randint(3, 5), cfl=0.2, steps=rng.randint(4, 12))


def _points(case):
    if case["kind"] == "run3d":
        return case["n0"] * case["n1"] * case["n2"]
    if case["kind"] == "ensemble":
        return sum(d["n"] for d in _instances(case, 0))
    return case["P"] * case["M"]


def work(case):
    """One read of the inputs and one write of the outputs; per update the
    operations of the central differences and the Euler step (a fused
    multiply-add counts two)."""
    N, w = _points(case), 8 if case["dtype"] == "f64" else 4
    if case["kind"] == "run3d":
        f = case["fields"]
        return {"bytes": 2 * N * f * w, "flops": N * f * case["steps"] * (16 if f == 1 else 24)}
    per = 9 if case["order"] == 2 else 16
    if case["kind"] == "adjoint":
        # u0, the target; u(T), the gradient; forward step, and the step's transpose
        return {"bytes": 4 * N * w, "flops": N * case["steps"] * 3 * per}
    per += 3 if case.get("forced") else 0
    return {"bytes": 2 * N * w, "flops": N * case["steps"] * per * (2 if case["comp"] else 1)}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _fourier(N, modes, seed):
    """sum_k k^-1 sin(k x + phi_k), seeded phases (an inverse real FFT)."""
    phi = torch.from_numpy(np.random.default_rng(seed).uniform(0.0, TWO_PI, size=modes)).cuda()
    k = torch.arange(1, modes + 1, device="cuda", dtype=torch.float64)
    X = torch.zeros(N // 2 + 1, dtype=torch.complex128, device="cuda")
    X[1:modes + 1] = torch.polar((N / 2.0) / k, phi - 0.5 * math.pi)
    return torch.fft.irfft(X, n=N)


def _field3(n, seed, kmax=32):
    """Random-phase field with E(k) ~ k^-5/3 up to |k| = kmax, max |u| = 1,
    shape (n2, n1, n0)."""
    n0, n1, n2 = n
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kx = torch.arange(0, n0 // 2 + 1, device="cuda", dtype=torch.float64)
    ky = torch.fft.fftfreq(n1, 1.0 / n1, device="cuda", dtype=torch.float64)
    kz = torch.fft.fftfreq(n2, 1.0 / n2, device="cuda", dtype=torch.float64)
    kk = (kz[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2).sqrt()
    amp = torch.where((kk >= 1) & (kk <= kmax), kk.clamp(min=1.0) ** (-11.0 / 6.0), torch.zeros_like(kk))
    ph = torch.rand(kk.shape, generator=g, device="cuda", dtype=torch.float64) * TWO_PI
    u = torch.fft.irfftn(torch.polar(amp, ph), s=(n2, n1, n0))
    return u / u.abs().max()


def _dt(umax, dx, nu, dim=1, cfl=0.2):
    return cfl * min(dx / umax, dx * dx / (2.0 * dim * nu))


def _instances(case, seed):
    """Travelling waves with seeded sizes, viscosities, speeds and delay bounds."""
    rng = np.random.default_rng(1000 + case["inst"])     # sizes and bounds: the case's
    sr = np.random.default_rng(seed)                     # viscosities and speeds: the seed's
    M, out = case["M"], []
    for _ in range(case["inst"]):
        n = max(M, int(round(2.0 ** rng.uniform(case["lo"], case["hi"]) / M)) * M)
        L = int(rng.integers(1, 4))
        nu = float(np.exp(sr.uniform(math.log(1e-3), math.log(1e-1))))
        c = float(sr.uniform(-0.5, 0.5))
        dx = TWO_PI / n
        a = min(0.5, 0.5 * nu / dx)
        out.append(dict(n=n, L=L, nu=nu, length=TWO_PI, origin=-math.pi, tanh_a=a, tanh_c=c, tanh_xc=0.0,
                        seed=int(sr.integers(0, 2 ** 62)), dt=_dt(abs(c) + a, dx, nu)))
    return out


def _per_point(inst, key):
    n = torch.tensor([d["n"] for d in inst], device="cuda")
    v = torch.tensor([float(d[key]) for d in inst], device="cuda", dtype=torch.float64)
    return torch.repeat_interleave(v, n)


def _waves(inst):
    n = torch.tensor([d["n"] for d in inst], device="cuda")
    first = torch.cumsum(n, 0) - n
    i = torch.arange(int(n.sum()), device="cuda") - torch.repeat_interleave(first, n)
    dx = torch.repeat_interleave(TWO_PI / n.double(), n)
    a, c, nu = (_per_point(inst, k) for k in ("tanh_a", "tanh_c", "nu"))
    return c - a * torch.tanh(a * (-math.pi + i * dx) / (2.0 * nu))


def _inputs(case, seed):
    """The run's fields and parameters (state in its own precision)."""
    tdt = torch.float64 if case["dtype"] == "f64" else torch.float32
    kind = case["kind"]
    if kind == "ensemble":
        inst = _instances(case, seed)
        return dict(inst=inst, u0=_waves(inst).to(tdt))
    if kind == "run3d":
        n = (case["n0"], case["n1"], case["n2"])
        f = case["fields"]
        u0 = torch.stack([_field3(n, seed * 8 + q).to(tdt) for q in range(f)])
        nu = 5e-3 if f == 1 else 2e-2
        kappa = [nu, nu, nu, 1e-2, 5e-2][:f] if f > 1 else [nu]
        dx = TWO_PI / max(n)                             # equal spacing on the three axes
        umax = 1.0 if f == 1 else 3.0
        return dict(n=n, u0=u0, kappa=kappa, length=tuple(dx * a for a in n),
                    dt=_dt(umax, dx, max(kappa), 3, case["cfl"]))
    N = case["P"] * case["M"]
    u = _fourier(N, min(64, max(4, N // 64)), seed)
    nu = {"adjoint": 0.01}.get(kind, 0.02 if N <= 65536 else 1e-3)
    d = dict(u0=u.to(tdt), nu=nu, dt=_dt(float(u.abs().max()), TWO_PI / N, nu), forcing=0.1 if case.get("forced") else 0.0)
    if kind == "adjoint":
        d["target"] = (u + 0.05 * _fourier(N, 8, seed + 77)).to(tdt)
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    d["case"], d["seed"] = case, seed
    flags = at.AT_FLAG_COMPENSATED if case.get("comp") else 0
    kind = case["kind"]
    if kind == "run1d":
        d["solver"] = at.Solver(case["P"] * case["M"], case["P"], case["order"], case["L"], d["nu"], d["dt"],
                                dtype=case["dtype"], forcing_amp=d["forcing"], seed=seed, flags=flags,
                                steps_per_pass=case["spp"])
    elif kind == "ensemble":
        most = max(i["L"] for i in d["inst"]) + 1
        d["solver"] = at.EnsembleSolver(d["inst"], case["M"], case["order"], dtype=case["dtype"], flags=flags,
                                        steps_per_pass=min(case["spp"], most), tile_subdomains=case["tile"])
    elif kind == "run3d":
        sub = (case["m0"], case["m1"], case["m2"])
        if case["fields"] == 1:
            d["solver"] = at.Solver3D(d["n"], sub, case["L"], d["kappa"][0], d["dt"], dtype=case["dtype"],
                                      length=d["length"], seed=seed, steps_per_pass=case["spp"])
        else:
            d["solver"] = at.System3D(d["n"], sub, case["L"], d["kappa"], d["dt"], dtype=case["dtype"],
                                      length=d["length"], seed=seed)
    else:
        d["u0"].requires_grad_(True)
        d["nu_t"] = torch.tensor(d["nu"], dtype=torch.float64, device="cuda", requires_grad=case["dtype"] == "f64")
    return d


def run(state):
    case = state["case"]
    if case["kind"] == "adjoint":
        u0, nu = state["u0"], state["nu_t"]
        uT = at.at_run(u0, nu, P=case["P"], order=case["order"], L=case["L"], dt=state["dt"], n_steps=case["steps"],
                       mode=at.AT_SEEDED, seed=state["seed"], interval=case["interval"])
        loss = ((uT - state["target"]) ** 2).sum()
        # (FP32 second differences at these spacings are rounding noise, so
        # only double-precision users ask for the viscosity's gradient)
        wrt = (u0, nu) if case["dtype"] == "f64" else (u0,)
        return [uT.detach(), *torch.autograd.grad(loss, wrt)]
    s = state["solver"]
    s.set_state(state["u0"])
    s.step(case["steps"], MODES[case["mode"]])
    return [s.state()]


# --------------------------------------------------------------------------
# the same runs in 64 bits
# --------------------------------------------------------------------------
_MASK = (1 << 64) - 1


def _i64(v):
    v &= _MASK
    return v - (1 << 64) if v >= 1 << 63 else v


def _shr(z, s):
    return (z >> s) & ((1 << (64 - s)) - 1)


def _delays(seed, ctr, L):
    """SplitMix64 draws at the counters, scaled to 0..L."""
    z = (ctr + 1) * _i64(0x9E3779B97F4A7C15) + _i64(seed)
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    z = z ^ _shr(z, 31)
    return (_shr(z, 32) * (L + 1)) >> 32


def _weights(k, s):
    """Extrapolation weights of the levels n-k-m, m = 0 .. s-1."""
    k = k.double()
    if s == 2:
        return [k + 1, -k]
    return [(k + 1) * (k + 2) / 2, -k * (k + 2), k * (k + 1) / 2]


def _rhs1(w, order, cA, cB):
    """dt (-u u_x + nu u_xx) from the stencil values w (offsets -R .. R)."""
    if order == 2:
        return cB * ((w[2] - w[1]) - (w[1] - w[0])) - cA * w[1] * (w[2] - w[0])
    a = 8 * (w[3] - w[1]) - (w[4] - w[0])
    b = 16 * ((w[3] - w[2]) - (w[2] - w[1])) - ((w[4] - w[2]) - (w[2] - w[0]))
    return cB * b - cA * w[2] * a


def _run64(u, case, dt, nu, forcing, seed, seeded):
    """The 1D AT run in FP64; u: [P, M]."""
    P, M = u.shape
    order, L = case["order"], case["L"]
    R, s = order // 2, order // 2 + 1
    N, dev = P * M, u.device
    dx = TWO_PI / N
    cA = dt / ((2 if order == 2 else 12) * dx)
    cB = nu * dt / ((1 if order == 2 else 12) * dx * dx)
    F = 0.0
    if forcing:
        F = dt * forcing * torch.sin(torch.arange(N, device=dev, dtype=torch.float64) * dx).view(P, M)
    left, right = [], []                   # last L + s levels' boundary words, newest first
    p = torch.arange(P, device=dev)
    for n in range(case["steps"]):
        left.insert(0, u[:, :R])
        right.insert(0, u[:, M - R:])
        del left[L + s:], right[L + s:]
        if seeded:
            kmax = max(0, n - s + 1)
            halo = []
            for f, hist, shift in ((0, right, 1), (1, left, -1)):
                k = _delays(seed, (n * P + p) * 2 + f, L).clamp(max=kmax)
                h = torch.stack([hist[min(i, len(hist) - 1)] for i in range(L + s)]).roll(shift, 1)
                halo.append(sum(wt[:, None] * h[k + m, p] for m, wt in enumerate(_weights(k, s))))
            lo, hi = halo
        else:
            lo, hi = right[0].roll(1, 0), left[0].roll(-1, 0)
        e = torch.cat([lo, u, hi], 1)
        u = u + (_rhs1([e[:, j:j + M] for j in range(2 * R + 1)], order, cA, cB) + F)
    return u


def _ensemble64(inst, u, case):
    n = torch.tensor([d["n"] for d in inst], device="cuda")
    last = torch.cumsum(n, 0) - 1
    first = last - n + 1
    g = {k: torch.tensor([float(d[k]) for d in inst], device="cuda", dtype=torch.float64)
         for k in ("nu", "dt", "tanh_a", "tanh_c")}
    dx = TWO_PI / n.double()
    cA = torch.repeat_interleave(g["dt"] / (2 * dx), n)
    cB = torch.repeat_interleave(g["nu"] * g["dt"] / (dx * dx), n)

    def wave(i, t):
        return g["tanh_c"] - g["tanh_a"] * torch.tanh(g["tanh_a"] * (-math.pi + i * dx - g["tanh_c"] * t) / (2 * g["nu"]))

    for lv in range(case["steps"]):
        lo, hi = u.roll(1), u.roll(-1)
        lo[first] = wave(-1, lv * g["dt"])
        hi[last] = wave(n, lv * g["dt"])
        u = u + _rhs1([lo, u, hi], 2, cA, cB)
    return u


def _run64_3d(d, case, seed, seeded):
    """The 3D run in FP64; fields (f, n2, n1, n0)."""
    q = d["u0"].double()
    f = q.shape[0]
    dt, L = d["dt"], case["L"]
    dx = [d["length"][a] / d["n"][a] for a in range(3)]
    sub = [case["m0"], case["m1"], case["m2"]]
    P = [d["n"][a] // sub[a] for a in range(3)]
    np_ = P[0] * P[1] * P[2]
    # [f, P2, m2, P1, m1, P0, m0]
    q = q.reshape(f, P[2], sub[2], P[1], sub[1], P[0], sub[0])
    axis = [(5, 6), (3, 4), (1, 2)]                      # (subdomain, point) dimensions of x, y, z
    sid = torch.arange(np_, device=q.device).view(P[2], P[1], P[0])
    hist = [[], []]                                      # [low faces, high faces] per level, newest first
    kap = [torch.tensor(d["kappa"], device=q.device, dtype=torch.float64).view(f, 1, 1, 1, 1, 1, 1)] * 3
    for n in range(case["steps"]):
        hist[0].insert(0, [q.narrow(axis[a][1], 0, 1).clone() for a in range(3)])
        hist[1].insert(0, [q.narrow(axis[a][1], sub[a] - 1, 1).clone() for a in range(3)])
        del hist[0][L + 2:], hist[1][L + 2:]
        inc = 0.0
        for a in range(3):
            sd, pd = axis[a]
            halo = []
            for side in (0, 1):
                h = [lv[a].roll(1 if side == 0 else -1, sd) for lv in hist[1 - side]]
                if not seeded:
                    halo.append(h[0])
                    continue
                k = _delays(seed, (n * np_ + sid) * 6 + 2 * a + side, L).clamp(max=max(0, n - 1))
                k = k.view(1, P[2], 1, P[1], 1, P[0], 1)
                v = torch.zeros_like(h[0])
                for kk in range(min(L, max(0, n - 1)) + 1):
                    e = h[0] if kk == 0 else (kk + 1) * h[kk] - kk * h[kk + 1]
                    v = torch.where(k == kk, e, v)
                halo.append(v)
            m = torch.cat([halo[0], q.narrow(pd, 0, sub[a] - 1)], pd)
            pl = torch.cat([q.narrow(pd, 1, sub[a] - 1), halo[1]], pd)
            vel = q if f == 1 else q[a:a + 1]
            inc = inc + kap[a] * (dt / dx[a] ** 2) * ((pl - q) - (q - m)) - dt / (2 * dx[a]) * vel * (pl - m)
        q = q + inc
    return q.reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    d = _inputs(case, seed)
    if kind == "ensemble":
        return [_ensemble64(d["inst"], d["u0"].double(), case)]
    if kind == "run3d":
        return [_run64_3d(d, case, seed, case["mode"] == "seeded")]
    u0 = d["u0"].double()
    shape = (case["P"], case["M"])
    if kind == "run1d":
        return [_run64(u0.view(shape), case, d["dt"], d["nu"], d["forcing"], seed, case["mode"] == "seeded").reshape(-1)]
    u0.requires_grad_(True)
    nu = torch.tensor(d["nu"], dtype=torch.float64, device="cuda", requires_grad=True)
    uT = _run64(u0.view(shape), case, d["dt"], nu, 0.0, seed, True).reshape(-1)
    loss = ((uT - d["target"].double()) ** 2).sum()
    return [uT.detach(), *torch.autograd.grad(loss, (u0, nu) if case["dtype"] == "f64" else (u0,))]
