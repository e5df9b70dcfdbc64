"""The work a program built on this library has it do, as cases that can be timed
and checked: whole studies (``simulate``, ``simulate_rrf``, ``Batch``, ``Server``)
and the steps of Algorithm 1 that a program may call on their own (the Latin
hypercube design, its correlation-reducing permutation, the reconstructed Wiener
increments and column moments).

``prepare`` draws the inputs from a seed (a seeded synthetic system of the
shape of the paper's case: symmetric B_ij ~ U[1, 8], G_ij ~ U[0, 0.3], diagonally
dominant, H ~ U[3, 10], D ~ U[1, 2], E ~ U[1, 1.1], Ornstein-Uhlenbeck
disturbances theta ~ U[0.5, 2], sigma ~ U[0.02, 0.1]), ``run`` makes one pass
through the public entry points, and ``exact`` restates the method in FP64 with
plain torch operations.
"""
import math
import types

import numpy as np
import torch

import paper_2007_03847_gb300 as fmc

LHS, SRS, SRS_EM = fmc.LHS, fmc.SRS, fmc.SRS_EM


# ---------------------------------------------------------------------------- cases


def listed():
    return [
        # one machine against an infinite bus, the smallest study: all latency
        dict(name="smib", kind="simulate", n=1, d=1, K=100, Nt=1000, dt=0.01, N=1000, precision="bf16x3"),
        # the paper's experiment: a generator trip at 1 s, the RMS frequency deviation
        # over 60 s, at the largest of its sample counts
        dict(name="trip_rms", kind="rrf", n=10, d=3, K=6, Nt=12000, dt=0.005, N=1000, precision="bf16x3"),
        # the benchmark: the 10-machine system shaped like the IEEE 39-bus case
        dict(name="ten_machines", kind="simulate", n=10, d=3, K=200, Nt=4000, dt=0.005, N=65536,
             precision="bf16x3"),
        # the same with the sample count of the precision study: the largest pass
        dict(name="ten_machines_large", kind="simulate", n=10, d=3, K=200, Nt=4000, dt=0.005, N=1048576,
             precision="bf16x3"),
        # the sampling comparison of one system: LHS, simple random sampling, the
        # traditional Monte Carlo (a normal per step) and the smooth random-ODE
        # forcing, as one batch; a ragged sample count
        dict(name="sampling_study", kind="arms", n=9, d=2, K=150, Nt=1000, dt=0.005, N=10007, precision="bf16x3"),
        # requests that arrive together at a server, small and uneven
        dict(name="serving", kind="serve", requests=8, n_hi=24, Nt_hi=1200, dt=0.005, N_lo=512, N_hi=4096,
             precision="bf16x3"),
        # systems too large for one thread per sample: 20 machines at full occupancy, 50
        # machines with fewer samples and eight disturbances
        dict(name="machines_20", kind="simulate", n=20, d=3, K=200, Nt=1000, dt=0.005, N=65536, precision="bf16x3"),
        dict(name="machines_50", kind="simulate", n=50, d=8, K=300, Nt=1000, dt=0.005, N=19001, precision="bf16x3"),
        # a batch of uneven scenarios in one captured graph
        dict(name="batch", kind="batch", count=8, n_hi=50, Nt_lo=500, Nt_hi=1500, dt=0.005, N_lo=1000, N_hi=16384,
             precision="bf16x3"),
        # the Latin hypercube design on its own: values and strata
        dict(name="design", kind="lhs", N=65536, M=600),
        # the design with the correlation-reducing permutation
        dict(name="design_rank", kind="rank", N=16384, M=600),
        # Wiener increments from given coefficients and their moments over the samples
        dict(name="increments", kind="paths", count=8192, d=3, K=200, Nt=2000, dt=0.005, precision="bf16x3"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["simulate", "simulate", "simulate", "large", "rrf", "arms", "serve", "batch", "lhs", "rank",
                       "paths"])
    prec = rng.choice(["bf16x3", "bf16x3", "bf16"])
    if kind == "simulate":
        n = rng.choice([1, rng.randint(4, 10), rng.randint(4, 10), rng.randint(11, 16)])
        return dict(kind=kind, n=n, d=1 if n == 1 else rng.randint(1, min(8, n)), K=rng.randint(50, 300),
                    Nt=_log(rng, 400, 4000), dt=0.005, N=_log(rng, 500, 262144), precision=prec,
                    heun=rng.random() < 0.2)
    if kind == "large":
        return dict(kind="simulate", n=rng.randint(17, 52), d=rng.randint(1, 8), K=rng.randint(50, 300),
                    Nt=rng.randint(300, 1000), dt=0.005, N=_log(rng, 1000, 65536), precision=prec)
    if kind == "rrf":
        return dict(kind=kind, n=rng.randint(4, 16), d=rng.randint(1, 4), K=rng.randint(6, 60),
                    Nt=_log(rng, 2000, 12000), dt=0.005, N=_log(rng, 20, 4000), precision=prec)
    if kind == "arms":
        return dict(kind=kind, n=rng.randint(4, 16), d=rng.randint(1, 4), K=rng.randint(50, 200),
                    Nt=rng.randint(400, 2000), dt=0.005, N=_log(rng, 1000, 32768), precision=prec)
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(2, 12), n_hi=rng.randint(10, 40), Nt_hi=rng.randint(1000, 2000),
                    dt=0.005, N_lo=256, N_hi=_log(rng, 1000, 8192), precision=prec)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 12), n_hi=rng.randint(10, 50), Nt_lo=400,
                    Nt_hi=rng.randint(800, 2000), dt=0.005, N_lo=1000, N_hi=_log(rng, 4000, 32768), precision=prec)
    if kind == "lhs":
        N, M = _log(rng, 1000, 1 << 20), rng.randint(50, 1200)
        return dict(kind=kind, N=N, M=max(20, min(M, (1 << 26) // N)))
    if kind == "rank":
        M = rng.randint(50, 800)
        return dict(kind=kind, N=max(M + 1, _log(rng, 1000, 40000)), M=M)
    return dict(kind="paths", count=_log(rng, 300, 12000), d=rng.randint(1, 4), K=rng.randint(20, 300),
                Nt=rng.randint(300, 2500), dt=0.005, precision=rng.choice([prec, "f32"]))


# ---------------------------------------------------------------------------- inputs


def _system(rng, n, d, **more):
    """A synthetic system and study, with the fields that the library reads."""
    if n == 1:
        V, X = 1.0, 0.5
        s = dict(G=np.zeros((1, 1)), B=np.array([[-1.0 / X]]), H=rng.uniform(4.0, 6.0, 1), D=rng.uniform(0.8, 1.2, 1),
                 E=np.array([1.1]), Pm=rng.uniform(0.6, 1.0, 1), theta=rng.uniform(0.8, 1.2, d),
                 sigma=rng.uniform(0.03, 0.07, d), inject=np.ones((1, d)), has_inf_bus=True, Ginf=np.zeros(1),
                 Binf=np.array([1.0 / X]), Vinf=V)
    else:
        B = np.triu(rng.uniform(1.0, 8.0, (n, n)), 1)
        G = np.triu(rng.uniform(0.0, 0.3, (n, n)), 1)
        B, G = B + B.T, G + G.T
        B[np.diag_indices(n)] = -B.sum(1) - rng.uniform(0.5, 2.0, n)
        G[np.diag_indices(n)] = G.sum(1) + rng.uniform(0.1, 0.5, n)
        E = rng.uniform(1.0, 1.1, n)
        inject = np.zeros((n, d))
        inject[rng.choice(n, size=d, replace=d > n), np.arange(d)] = 1.0
        s = dict(G=G, B=B, H=rng.uniform(3.0, 10.0, n), D=rng.uniform(1.0, 2.0, n), E=E,
                 Pm=E * (G @ E) + rng.uniform(-1.0, 2.0, n), theta=rng.uniform(0.5, 2.0, d),
                 sigma=rng.uniform(0.02, 0.1, d), inject=inject, has_inf_bus=False, Ginf=None, Binf=None, Vinf=1.0)
    s.update(n=n, d=d, omega_s=2.0 * math.pi * 50.0, seed=int(rng.integers(1 << 62)), sampling=LHS,
             forcing=fmc.FORCING_INCREMENTS, event_machine=None, event_time=0.0, event_dpm=0.0)
    s.update(more)
    s["T"] = s["Nt"] * s["dt"]
    return types.SimpleNamespace(**s)


def _scenarios(case, seed):
    rng = np.random.default_rng([seed, 7])
    k = case["kind"]
    if k in ("simulate", "rrf"):
        more = {x: case[x] for x in ("K", "Nt", "dt", "N")}
        if k == "rrf":
            sc = _system(rng, case["n"], case["d"], **more)
            sc.event_machine = int(rng.integers(case["n"]))
            sc.event_time, sc.event_dpm = 1.0, -0.5
            return [sc]
        return [_system(rng, case["n"], case["d"], **more)]
    if k == "arms":
        one = _system(rng, case["n"], case["d"], **{x: case[x] for x in ("K", "Nt", "dt", "N")})
        arms = [types.SimpleNamespace(**vars(one)) for _ in range(4)]
        arms[1].sampling, arms[2].sampling, arms[3].forcing = SRS, SRS_EM, fmc.FORCING_SMOOTH
        return arms
    # batch, serve: uneven scenarios; the sizes are the case's own, the systems the seed's
    count = case["count"] if k == "batch" else case["requests"]
    sizes = np.random.default_rng([count, case["n_hi"], case["N_hi"], case["Nt_hi"]])
    out = []
    for _ in range(count):
        n, d, K = (int(sizes.integers(a, b + 1)) for a, b in ((4, case["n_hi"]), (1, 8), (50, 300)))
        Nt = int(sizes.integers(case.get("Nt_lo", case["Nt_hi"] // 2), case["Nt_hi"] + 1))
        N = int(round(math.exp(sizes.uniform(math.log(case["N_lo"]), math.log(case["N_hi"])))))
        out.append(_system(rng, n, d, K=K, Nt=Nt, dt=case["dt"], N=N))
    return out


def prepare(case, seed):
    k = case["kind"]
    if k in ("lhs", "rank"):
        return dict(case=case, seed=int(np.random.default_rng([seed, 3]).integers(1 << 62)))
    if k == "paths":
        g = torch.Generator(device="cuda").manual_seed(seed)
        z = torch.randn(case["count"], case["d"] * case["K"], device="cuda", generator=g)
        return dict(case=case, zeta=z)
    scs = _scenarios(case, seed)
    state = dict(case=case, scs=scs)
    if k in ("arms", "batch"):
        state["batch"] = fmc.Batch(scs, precision=case["precision"])
    if k == "serve":
        state["server"] = fmc.Server(slots=4, mem_budget_bytes=32 << 30)
    return state


# ---------------------------------------------------------------------------- a pass


def run(state):
    case, k = state["case"], state["case"]["kind"]
    if k == "simulate":
        return fmc.simulate(state["scs"][0], precision=case["precision"],
                            integrator=fmc.HEUN if case.get("heun") else fmc.RK4)
    if k == "rrf":
        return fmc.simulate_rrf(state["scs"][0], precision=case["precision"])
    if k in ("arms", "batch"):
        return state["batch"].launch()
    if k == "serve":
        srv = state["server"]
        handles = [srv.submit(sc, precision=case["precision"]) for sc in state["scs"]]
        out = []
        for h in handles:
            res, mean, var = srv.wait(h)
            out.append((res["status"], mean, var))
        return out
    if k == "lhs":
        strata = torch.empty(case["M"], case["N"], dtype=torch.int32, device="cuda")
        return fmc.lhs_sample(state["seed"], case["N"], case["M"], strata=strata)
    if k == "rank":
        return fmc.lhs_decorrelate(state["seed"], case["N"], case["M"])
    dW = fmc.kle_reconstruct(state["zeta"], case["d"], case["K"], case["Nt"] * case["dt"], case["dt"],
                             precision=case["precision"])
    return (dW,) + tuple(fmc.moments(dW))


def work(case):
    k = case["kind"]
    if k in ("lhs", "rank"):
        # a value and a stratum written per entry; the permutation of the rank form
        # needs the product R Q^-T and the correlation matrix
        N, M = case["N"], case["M"]
        return dict(bytes=8.0 * N * M, flops=(3.0 * N * M * M if k == "rank" else 0.0))
    if k == "paths":
        c, d, K, Nt = case["count"], case["d"], case["K"], case["Nt"]
        return dict(bytes=4.0 * c * d * K + 4.0 * c * d * Nt + 16.0 * d * Nt, flops=2.0 * c * d * K * Nt)
    b = f = 0.0
    for sc in _scenarios(case, 1):
        # per sample, step, stage and machine the network sums take 4 n products and the
        # rest about 8; the moments are written once, the system read once
        b += 32.0 * sc.n * (sc.Nt + 1) + 16.0 * sc.n * sc.n
        f += 2.0 * sc.N * sc.Nt * sc.n * (16.0 * sc.n + 32.0) + 2.0 * sc.N * sc.d * sc.Nt * (
            0 if sc.sampling == SRS_EM else sc.K)
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------------------- the method in FP64

_DEV = "cuda" if torch.cuda.is_available() else "cpu"
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, key):
    """Words of Philox4x32-10 (int64 tensors or ints holding 32-bit values)."""
    k0, k1 = key & _M32, (key >> 32) & _M32
    for _ in range(10):
        # (a 64-bit product wraps; its high word is masked after the shift)
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _zero(x):
    return torch.zeros_like(x)


def _strata(key, N, dims):
    """pi_i(k) for all samples and the given dimensions: int64 [N, len(dims)]."""
    h = max(1, (max(N - 1, 0).bit_length() + 1) // 2)
    mask = (1 << h) - 1
    k = torch.arange(N, device=_DEV)[:, None].expand(N, len(dims)).reshape(-1)
    dim = dims[None, :].expand(N, len(dims)).reshape(-1)
    y = k.clone()
    todo = torch.arange(y.numel(), device=_DEV)
    while todo.numel():
        v, dd = y[todo], dim[todo]
        L, R = (v >> h) & mask, v & mask
        for r in range(6):
            o = _philox(R, dd, _zero(R) + (1 + r), _zero(R), key)[0]
            L, R = R, L ^ (o & mask)
        v = (L << h) | R
        y[todo] = v
        todo = todo[v >= N]
    return y.reshape(N, len(dims))


def _uniforms(key, N, dims):
    k = torch.arange(N, device=_DEV)[:, None].expand(N, len(dims))
    dd = dims[None, :].expand(N, len(dims))
    return (_philox(k, dd, _zero(k), _zero(k), key)[0].double() + 0.5) / 4294967296.0


def _normal(lower, upper):
    """Phi^-1 of a probability given with its complement (both tails keep their digits)."""
    return torch.where(lower < 0.5, torch.special.ndtri(lower), -torch.special.ndtri(upper))


def _design(key, N, M, sampling):
    """The design's values [N, M] in FP64, and its strata."""
    z = torch.empty(N, M, dtype=torch.float64, device=_DEV)
    st = torch.empty(N, M, dtype=torch.int64, device=_DEV)
    step = max(1, (1 << 22) // N)
    for a in range(0, M, step):
        dims = torch.arange(a, min(M, a + step), device=_DEV)
        u = _uniforms(key, N, dims)
        if sampling == SRS:
            z[:, a:a + step] = _normal(u, 1.0 - u)
            continue
        s = _strata(key, N, dims)
        st[:, a:a + step] = s
        z[:, a:a + step] = _normal((s + u) / N, ((N - 1 - s) + (1.0 - u)) / N)
    return z, st


def _basis(K, T, Nt):
    k = torch.arange(K, device=_DEV, dtype=torch.float64)[:, None] * 2 + 1
    n = torch.arange(Nt, device=_DEV, dtype=torch.float64)[None, :] * 2 + 1
    ang = torch.remainder(k * n, 8.0 * Nt) * (math.pi / (4.0 * Nt))
    c = 2.0 * math.sqrt(2.0 * T) / (k * math.pi)
    return 2.0 * c * torch.cos(ang) * torch.sin(math.pi * k / (4.0 * Nt))


def _forcing(K, T, Nt):
    k = torch.arange(K, device=_DEV, dtype=torch.float64)[:, None] * 2 + 1
    j = torch.arange(2 * Nt + 1, device=_DEV, dtype=torch.float64)[None, :]
    return math.sqrt(2.0 / T) * torch.cos(torch.remainder(k * j, 8.0 * Nt) * (math.pi / (4.0 * Nt)))


def _equilibrium(sc):
    """delta* and the balanced mechanical powers (numpy, Newton from a flat start)."""
    n, first = sc.n, (0 if sc.has_inf_bus else 1)
    G, B, E = sc.G, sc.B, sc.E
    delta, Pm = np.zeros(n), np.array(sc.Pm, dtype=np.float64)
    for _ in range(100):
        a, b = E * np.cos(delta), E * np.sin(delta)
        u, v = G @ a - B @ b, G @ b + B @ a
        Pe = a * u + b * v
        J = G * (np.outer(b, a) - np.outer(a, b)) - B * (np.outer(a, a) + np.outer(b, b))
        J[np.diag_indices(n)] = a * v - b * u - np.diag(B) * (a * a + b * b)
        if sc.has_inf_bus:
            Pe = Pe + sc.Vinf * (sc.Ginf * a + sc.Binf * b)
            J[np.diag_indices(n)] += sc.Vinf * (sc.Binf * a - sc.Ginf * b)
        F = (Pm - Pe)[first:]
        if F.size == 0 or np.max(np.abs(F)) < 1e-12:
            break
        delta[first:] += np.linalg.solve(J[first:, first:], F)
    if first:
        Pm[0] = Pe[0]
    return delta, Pm


def _study(sc, rrf=False, heun=False):
    """Mean and variance [Nt+1, 2n] (and E, Var of the RMS frequency deviation)."""
    f64 = dict(dtype=torch.float64, device=_DEV)
    n, d, N, Nt, dt = sc.n, sc.d, sc.N, sc.Nt, sc.dt
    t = lambda x: torch.as_tensor(np.asarray(x, dtype=np.float64), **f64)  # noqa: E731
    delta0, Pm = _equilibrium(sc)
    E, i2h, D, inj = t(sc.E), t(1.0 / (2.0 * sc.H)), t(sc.D), t(sc.inject)
    # [a b] -> [u v] of the network's product form
    net = torch.cat([torch.cat([t(sc.G).T, t(sc.B).T], 1), torch.cat([-t(sc.B).T, t(sc.G).T], 1)], 0).contiguous()
    Pm = t(Pm)
    delta = t(delta0).expand(N, n).clone()
    w = torch.zeros(N, n, **f64)
    x = torch.zeros(N, d, **f64)
    mean = torch.zeros(Nt + 1, 2 * n, **f64)
    var = torch.zeros(Nt + 1, 2 * n, **f64)
    mean[0, :n] = t(delta0)
    if N == 1:
        var[:] = math.nan
    smooth = sc.forcing == fmc.FORCING_SMOOTH
    theta, sigma = t(sc.theta), t(sc.sigma)
    hw = t(sc.H / np.sum(sc.H))
    racc = torch.zeros(N, **f64)
    ev_step = int(round(sc.event_time / dt)) if sc.event_machine is not None else Nt + 1
    if sc.sampling != SRS_EM:
        z = _design(sc.seed, N, d * sc.K, sc.sampling)[0].reshape(N * d, sc.K)
        phi = _forcing(sc.K, sc.T, Nt) if smooth else _basis(sc.K, sc.T, Nt)
    ks = torch.arange(N, device=_DEV)

    def rate(dl, om, xs, ev):
        a, b = E * torch.cos(dl), E * torch.sin(dl)
        uv = torch.cat([a, b], 1) @ net
        Pe = a * uv[:, :n] + b * uv[:, n:]
        if sc.has_inf_bus:
            Pe = Pe + sc.Vinf * (t(sc.Ginf) * a + t(sc.Binf) * b)
        kw = (Pm + xs @ inj.T - Pe - D * om) * i2h
        if ev:
            kw[:, sc.event_machine] += sc.event_dpm * i2h[sc.event_machine]
        return sc.omega_s * om, kw

    def collect(row, dl, om):
        both = torch.cat([dl, om], 1)
        if N > 1:
            var[row], mean[row] = torch.var_mean(both, 0)
        else:
            mean[row] = both[0]
        if rrf:
            racc.add_((om @ hw) ** 2)

    block = max(1, min(Nt, (1 << 27) // (N * d)))
    for n0 in range(0, Nt, block):
        m = min(block, Nt - n0)
        # increments (or the forcing at the half steps) of this block: [m or 2m+1, N, d]
        if sc.sampling == SRS_EM:
            inc = torch.empty(m, N, d, **f64)
            for s in range(m):
                for q in range(d):
                    r = _philox(ks, _zero(ks) + (n0 + s), _zero(ks) + 256, _zero(ks) + q // 4, sc.seed)[q % 4]
                    u = (r.double() + 0.5) / 4294967296.0
                    inc[s, :, q] = math.sqrt(dt) * _normal(u, 1.0 - u)
        else:
            cols = phi[:, 2 * n0:2 * (n0 + m) + 1] if smooth else phi[:, n0:n0 + m]
            inc = (z @ cols).T.reshape(cols.shape[1], N, d)
        for s in range(m):
            ev = n0 + s >= ev_step
            if smooth:
                f0, fh, f1 = inc[2 * s], inc[2 * s + 1], inc[2 * s + 2]
                k1 = sigma * f0 - theta * x
                x2 = x + 0.5 * dt * k1
                k2 = sigma * fh - theta * x2
                x3 = x + 0.5 * dt * k2
                k3 = sigma * fh - theta * x3
                x4 = x + dt * k3
                k4 = sigma * f1 - theta * x4
                stages = (x, x2, x3, x4)
                x = x + dt / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
            else:
                x1 = (1.0 - theta * dt) * x + sigma * inc[s]
                mid = 0.5 * (x + x1)
                stages = (x, mid, mid, x1)
                x = x1
            a1, b1 = rate(delta, w, stages[0], ev)
            if heun:
                a2, b2 = rate(delta + dt * a1, w + dt * b1, stages[3], ev)
                delta, w = delta + 0.5 * dt * (a1 + a2), w + 0.5 * dt * (b1 + b2)
                collect(n0 + s + 1, delta, w)
                continue
            a2, b2 = rate(delta + 0.5 * dt * a1, w + 0.5 * dt * b1, stages[1], ev)
            a3, b3 = rate(delta + 0.5 * dt * a2, w + 0.5 * dt * b2, stages[2], ev)
            a4, b4 = rate(delta + dt * a3, w + dt * b3, stages[3], ev)
            delta = delta + dt / 6.0 * (a1 + 2 * a2 + 2 * a3 + a4)
            w = w + dt / 6.0 * (b1 + 2 * b2 + 2 * b3 + b4)
            collect(n0 + s + 1, delta, w)
    if not rrf:
        return mean, var
    r = torch.sqrt(racc / Nt)
    return torch.stack([r.mean(), r.var() if N > 1 else r.new_tensor(math.nan)]), mean, var


def _seconds(sc):
    """About what _study takes on a GPU: launches, or FP64 work."""
    step = max(1.5e-3, 4 * sc.N * sc.n * (2.5e-10 + 1.2e-11 * sc.n))
    if sc.sampling == SRS_EM:
        step += 2.5e-3 * sc.d
    return sc.Nt * step


def _rank(key, N, M):
    """The correlation-reducing permutation (rank method): values and strata."""
    s = torch.arange(N, device=_DEV, dtype=torch.float64)
    score = _normal((s + 1) / (N + 1), (N - s) / (N + 1))
    score = score - score.mean()
    dims = torch.arange(M, device=_DEV)
    R = score[_strata(key, N, dims)]
    C = R.T @ R
    dg = torch.sqrt(torch.diagonal(C))
    Q = torch.linalg.cholesky(C / (dg[:, None] * dg[None, :]))
    Rs = torch.linalg.solve_triangular(Q, R.T, upper=False)  # [M, N]: R* transposed
    order = torch.sort(Rs, dim=1, stable=True).indices
    new = torch.empty_like(order)
    new.scatter_(1, order, torch.arange(N, device=_DEV).expand(M, N))
    st = new.T
    u = _uniforms(key, N, dims)
    return _normal((st + u) / N, ((N - 1 - st) + (1.0 - u)) / N)


def exact(case, seed):
    k = case["kind"]
    if k == "lhs":
        if case["N"] * case["M"] > 1 << 26:
            return None
        key = int(np.random.default_rng([seed, 3]).integers(1 << 62))
        return _design(key, case["N"], case["M"], LHS)[0], None
    if k == "rank":
        key = int(np.random.default_rng([seed, 3]).integers(1 << 62))
        return _rank(key, case["N"], case["M"]), None
    if k == "paths":
        z = prepare(case, seed)["zeta"].double().reshape(-1, case["K"])
        dW = (z @ _basis(case["K"], case["Nt"] * case["dt"], case["Nt"])).reshape(case["count"], case["d"], case["Nt"])
        var, mean = torch.var_mean(dW, 0)
        return dW, mean, var
    scs = _scenarios(case, seed)
    if k in ("simulate", "rrf"):
        return _study(scs[0], k == "rrf", bool(case.get("heun"))) if _seconds(scs[0]) < 25 else None
    left, got = 18.0, []
    for sc in scs:
        left -= _seconds(sc)
        got.append(_study(sc) if left > 0 else (None, None))
    if k == "serve":
        return [(None, m, v) for m, v in got]
    return [m for m, _ in got], [v for _, v in got]
