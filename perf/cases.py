"""The workloads by which the speed of this library is measured.

Each case is one call (or the few calls) a user's program makes through the
package's public entry points: HMC trajectories, CG solves, observables, the
standalone Q applies and the batched multi-chain engine, on lattices of the
sizes that the configurations, tests and benchmark of this repository name
(d = 1 chains, d = 3 lattices of N_x = 8 .. 32), in both precisions.

``exact`` recomputes the outputs in FP64 with plain torch (Eqs. (7)-(12): the
operator by torch.roll, textbook CG with residual replacement, leapfrog, the
Philox streams by numpy's generator), without this package's code.
"""
import math

import numpy as np
import torch

import paper_1007_3432_gb300 as hh
from paper_1007_3432_gb300 import binding

HOP, DTAU, A_HS = 1.0, 0.05, 0.5
H = HOP * DTAU


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # The smallest chains: a few thousand sites, where a CG iteration is
        # all latency.  Heatbath, 6 forces of 2 pseudofermions, Metropolis.
        dict(name="hmc_d1_32x64_fp64", kind="hmc", d=1, nx=32, ntau=64, precision="fp64", n_md=5, dt=0.02),
        # The same for the smallest d = 3 lattice of the batch range.
        dict(name="hmc_d3_8x40_fp64", kind="hmc", d=3, nx=8, ntau=40, precision="fp64", n_md=4, dt=0.02),
        # An HMC step of an ordinary d = 3 lattice in mixed precision.
        dict(name="hmc_d3_12x64_mixed", kind="hmc", d=3, nx=12, ntau=64, precision="mixed", n_md=3, dt=0.02),
        # Solves of measurement programs: two sources on a long d = 1 chain in
        # FP64, an odd length in mixed precision (no vector width divides it).
        dict(name="solve_d1_1024x128_fp64", kind="solve", d=1, nx=1024, ntau=128, precision="fp64", n_rhs=2),
        dict(name="solve_d1_731x96_mixed", kind="solve", d=1, nx=731, ntau=96, precision="mixed", n_rhs=2),
        # d = 3 lattices of the paper's study (N_x = 8 .. 20), one and two sources.
        dict(name="solve_d3_16x64_mixed", kind="solve", d=3, nx=16, ntau=64, precision="mixed", n_rhs=1),
        dict(name="solve_d3_20x96_mixed", kind="solve", d=3, nx=20, ntau=96, precision="mixed", n_rhs=2),
        # The largest lattice of the benchmark: the vectors stream from HBM.
        dict(name="solve_d3_32x128_mixed", kind="solve", d=3, nx=32, ntau=128, precision="mixed", n_rhs=2),
        # The preconditioned solver, as long d = 1 chains are served.
        dict(name="pcg_d1_256x256_fp64", kind="solve", d=1, nx=256, ntau=256, precision="fp64", n_rhs=2, cheb=8),
        # Measurement of the occupation with the exact-block form of M.
        dict(name="observables_d3_10x48_block", kind="observables", d=3, nx=10, ntau=48, precision="fp64",
             order=1, n_noise=4),
        # Q on many vectors that share a field (block Krylov, eigensolvers).
        dict(name="apply_d3_32x128_16vec_f32", kind="apply", d=3, nx=32, ntau=128, dtype="f32", n_vec=16),
        # Independent chains of uneven volumes in the batched engine.
        dict(name="batch_d3_10chains_mixed", kind="batch", precision="mixed", chains=10, nx_min=8, nx_max=16,
             ntau_min=40, ntau_max=96, n_rhs=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("hmc", "hmc", "solve", "solve", "solve", "solve", "pcg", "observables", "apply", "apply",
                       "batch"))
    d = rng.choice((1, 3))
    if kind == "hmc":
        nx, ntau = (_log_int(rng, 16, 256), rng.randrange(24, 81)) if d == 1 else (rng.randint(4, 14), rng.randrange(24, 65))
        return dict(kind="hmc", d=d, nx=nx, ntau=ntau, precision=rng.choice(("fp64", "mixed")), n_md=rng.randint(2, 4),
                    dt=0.02)
    if kind == "solve":
        precision = rng.choice(("fp64", "mixed"))
        if d == 1:
            nx, ntau = _log_int(rng, 24, 2048), rng.randrange(32, 113)
        else:
            nx, ntau = rng.randint(4, 18 if precision == "fp64" else 24), rng.randrange(24, 97)
        return dict(kind="solve", d=d, nx=nx, ntau=ntau, precision=precision, n_rhs=rng.randint(1, 3))
    if kind == "pcg":
        return dict(kind="solve", d=1, nx=_log_int(rng, 64, 512), ntau=rng.randrange(64, 257), precision="fp64",
                    n_rhs=rng.randint(1, 2), cheb=8)
    if kind == "observables":
        nx, ntau = (_log_int(rng, 32, 512), rng.randrange(24, 81)) if d == 1 else (rng.randint(4, 12), rng.randrange(24, 65))
        return dict(kind="observables", d=d, nx=nx, ntau=ntau, precision=rng.choice(("fp64", "mixed")),
                    order=rng.choice((0, 1)), n_noise=rng.choice((2, 4, 8)))
    if kind == "apply":
        dtype = rng.choice(("f32", "f64"))
        if d == 1:
            nx, ntau = _log_int(rng, 32, 2048), rng.randrange(32, 513)
        else:
            nx, ntau = rng.randint(6, 32), rng.randrange(16, 129)
        return dict(kind="apply", d=d, nx=nx, ntau=ntau, dtype=dtype, n_vec=rng.choice((1, 1, 2, 4, 8)))
    return dict(kind="batch", precision=rng.choice(("fp64", "mixed")), chains=rng.randint(2, 8), nx_min=rng.randint(6, 8),
                nx_max=rng.randint(9, 12), ntau_min=40, ntau_max=rng.randrange(41, 81), n_rhs=rng.randint(1, 2))


def _sites(case):
    return case["nx"] ** case["d"] * case["ntau"]


def _chains(case):
    """Lattices (N_x, N_tau) of a batch: spread over its ranges, uneven volumes."""
    n = case["chains"]
    out = []
    for j in range(n):
        f = j / max(1, n - 1)
        g = (j * 0.618034) % 1.0
        out.append((case["nx_min"] + int(round(f * (case["nx_max"] - case["nx_min"]))),
                    case["ntau_min"] + int(round(g * (case["ntau_max"] - case["ntau_min"])))))
    return out


# ---------------------------------------------------------------------------
# States and passes
# ---------------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) + 1)


def _field(n, gen):
    """A hot-start field: i.i.d. uniform on [-pi, pi)."""
    return (torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) * 2.0 - 1.0) * math.pi


def _inputs(case, seed):
    """Field and vectors of a case (device tensors), from the seed alone."""
    gen = _generator(seed)
    n = _sites(case)
    out = {"sigma": _field(n, gen)}
    if case["kind"] == "solve":
        out["b"] = torch.randn(case["n_rhs"], n, dtype=torch.float64, device="cuda", generator=gen)
    elif case["kind"] == "apply":
        t = torch.float32 if case["dtype"] == "f32" else torch.float64
        out["x"] = torch.randn(case["n_vec"], n, dtype=torch.float64, device="cuda", generator=gen).to(t)
    return out


def _batch_inputs(case, seed):
    """Host arrays of a batch's requests, as a program submits them."""
    out = []
    for j, (nx, ntau) in enumerate(_chains(case)):
        n = nx ** 3 * ntau
        g = np.random.Generator(np.random.Philox(key=[int(seed) + 1, j]))
        out.append((nx, ntau, g.uniform(-math.pi, math.pi, n), g.standard_normal((case["n_rhs"], n))))
    return out


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case}
    if kind == "batch":
        reqs = []
        for nx, ntau, sigma, b in _batch_inputs(case, seed):
            out = np.zeros_like(b)
            req = binding.make_request(binding.HH_REQ_SOLVE, 3, nx, ntau, sigma=sigma, b=b, out=out,
                                       precision=case["precision"], n_pf=case["n_rhs"], t=HOP, dtau=DTAU, A=A_HS)
            reqs.append((req, (sigma, b, out)))
        state["reqs"] = reqs
        state["batch"] = binding.Batch(max_slots=64, hbm_budget_bytes=1 << 30)
        return state
    state.update(_inputs(case, seed))
    kw = dict(t=HOP, dtau=DTAU, A=A_HS, seed=int(seed) & 0xFFFFFFFF)
    if kind != "apply":
        kw["precision"] = case["precision"]
    if case.get("cheb"):
        kw.update(cheb_degree=case["cheb"], cheb_eps=1e-4)
    if case.get("order"):
        kw["link_order"] = case["order"]
    state["ctx"] = hh.Context(case["d"], case["nx"], case["ntau"], **kw)
    state["ctx"].set_field(state["sigma"])
    if kind == "solve":
        state["x"] = torch.zeros_like(state["b"])
    elif kind == "apply":
        state["y"] = torch.empty_like(state["x"])
    elif kind == "hmc":
        state["out"] = torch.empty_like(state["sigma"])
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        state["ctx"].solve(state["b"], state["x"], case["n_rhs"])
        return {"x": state["x"]}
    if kind == "apply":
        if case["n_vec"] == 1:
            state["ctx"].apply(binding.HH_OP_MTM, state["x"][0], state["y"][0])
        else:
            state["ctx"].apply_multi(binding.HH_OP_MTM, state["x"], state["y"], case["n_vec"])
        return {"y": state["y"]}
    if kind == "hmc":
        # One trajectory from a stored configuration.
        ctx = state["ctx"]
        ctx.set_field(state["sigma"])
        info = ctx.trajectory(case["n_md"], case["dt"], 0)
        ctx.get_field(state["out"])
        return {"sigma": state["out"], "H0": np.float64(info["H0"]), "H1": np.float64(info["H1"]),
                "accepted": int(info["accepted"])}
    if kind == "observables":
        o = state["ctx"].observables(case["n_noise"], 0)
        return {k: np.float64(o[k]) for k in ("trace_Minv", "trace_err", "one_minus_g_sq", "mean_sin", "mean_sin2")}
    batch = state["batch"]
    for req, keep in state["reqs"]:
        batch.submit(req, keep=keep)
    done = batch.run_until_idle()
    return {"x": [keep[2] for _, keep in state["reqs"]], "failed": sum(1 for r in done if r["status"] != 0)}


# ---------------------------------------------------------------------------
# What a pass cannot do without, and how close two correct passes are
# ---------------------------------------------------------------------------

def _steps(d, ntau):
    """CG steps of a hot lattice of this temporal extent to a true residual of
    1e-10 (a fit to measured counts, for the operation count only)."""
    return 1300.0 * (ntau / 40.0) ** 1.53 if d == 3 else 2000.0 * (ntau / 64.0) ** 1.9 + 2100.0


def _solve_work(d, nx, ntau, n_rhs):
    n = nx ** d * ntau
    # Per site and step: 2d + 3 operations in each of M and M^T, 10 in the
    # vector updates and dot products; the preconditioned solve applies Q about
    # as often as the plain one takes steps.
    flops = n_rhs * n * _steps(d, ntau) * (2 * (2 * d + 3) + 10)
    return {"bytes": n * (8.0 + 16.0 * n_rhs), "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        ws = [_solve_work(3, nx, ntau, case["n_rhs"]) for nx, ntau in _chains(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    d, nx, ntau, n = case["d"], case["nx"], case["ntau"], _sites(case)
    if kind == "solve":
        return _solve_work(d, nx, ntau, case["n_rhs"])
    if kind == "apply":
        w = 4 if case["dtype"] == "f32" else 8
        return {"bytes": float(w * n * (2 * case["n_vec"] + 1)), "flops": float(n * case["n_vec"] * 2 * (2 * d + 3))}
    if kind == "hmc":
        w = _solve_work(d, nx, ntau, 2)
        return {"bytes": 16.0 * n, "flops": w["flops"] * (case["n_md"] + 1)}
    w = _solve_work(d, nx, ntau, case["n_noise"])
    # Five numbers come back; the field is what is read.
    return {"bytes": 8.0 * n, "flops": w["flops"]}


def tolerance(case):
    """About four times the distance measured against exact()."""
    kind = case["kind"]
    if kind == "apply":
        return {"rel": 2e-7} if case["dtype"] == "f32" else {"rel": 4e-16}
    if kind == "hmc":
        return {"rel": 2e-10, "max": 1e-7}
    if kind == "observables":
        return {"rel": 2e-8, "max": 2e-8}
    # Solutions with a true relative residual of 1e-10: 1e-10 to 2.6e-10 from
    # the exact ones.
    return {"rel": 2e-9, "max": 1e-6}


# ---------------------------------------------------------------------------
# The same in plain FP64 torch
# ---------------------------------------------------------------------------

class _Lattice:
    """M, M^T and Q of Eq. (10) on arrays (..., tau, z, y, x)."""

    def __init__(self, d, nx, ntau, sigma, order=0):
        self.shape = (ntau,) + (nx,) * d
        self.axes = tuple(range(-d, 0))
        self.tax = -d - 1
        self.order = order
        self.sigma = sigma.reshape(self.shape)
        self.sign = torch.full((ntau,) + (1,) * d, -1.0, dtype=torch.float64, device=sigma.device)
        self.sign[-1] = 1.0
        self.L = self.sign * (1.0 + A_HS * torch.sin(self.sigma))

    def hop(self, v):
        s = torch.zeros_like(v)
        for a in self.axes:
            s = s + torch.roll(v, 1, a) + torch.roll(v, -1, a)
        return s

    def block(self, v):
        """e^{hH} to the form's order."""
        s = self.hop(v)
        e = v + H * s
        return e + 0.5 * H * H * self.hop(s) if self.order == 2 else e

    def M(self, v):
        if self.order:
            return v + torch.roll(self.block(self.L * v), 1, self.tax)
        return v - H * self.hop(v) + torch.roll(self.L * v, 1, self.tax)

    def MT(self, v):
        if self.order:
            return v + self.L * torch.roll(self.block(v), -1, self.tax)
        return v - H * self.hop(v) + self.L * torch.roll(v, -1, self.tax)

    def solve(self, b, tol=1e-14):
        """Q x = b for each leading index of b: CG from zero, restarted from
        the true residual until that stops falling."""
        x = torch.zeros_like(b)
        dims = tuple(range(1, b.dim()))

        def dot(u, v):
            return (u * v).sum(dims, keepdim=True)

        bb = dot(b, b)
        best = math.inf
        for _ in range(6):
            r = b - self.MT(self.M(x))
            rr = dot(r, r)
            now = float((rr / bb).max())
            if now <= tol * tol or now > 0.25 * best:
                break
            best = now
            start = rr.clone()
            p = r.clone()
            for it in range(60000):
                t = self.M(p)
                alpha = rr / dot(t, t).clamp_min(1e-300)
                x = x + alpha * p
                r = r - alpha * self.MT(t)
                new = dot(r, r)
                p = r + (new / rr.clamp_min(1e-300)) * p
                rr = new
                if it % 64 == 63 and bool((rr <= torch.maximum(1e-12 * start, 0.25 * tol * tol * bb)).all()):
                    break
        return x


def _philox(n_blocks, tag, a, traj, chain, seed):
    """Words (n_blocks, 4) of Philox4x64-10 with counter (block, tag | a << 8,
    traj, chain) and key (seed, 0); numpy's generator steps the counter first."""
    c = (tag | (a << 8)) << 64 | traj << 128 | chain << 192
    c = (c - 1) % (1 << 256)
    words = np.array([(c >> (64 * j)) & ((1 << 64) - 1) for j in range(4)], dtype=np.uint64)
    return np.random.Philox(counter=words, key=np.array([seed, 0], dtype=np.uint64)).random_raw(4 * n_blocks).reshape(-1, 4)


def _u53(w):
    return (w >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _gaussian(n, tag, a, seed):
    w = _philox((n + 3) // 4, tag, a, 0, 0, seed)
    out = np.empty((w.shape[0], 4))
    for j in (0, 2):
        r = np.sqrt(-2.0 * np.log(1.0 - _u53(w[:, j])))
        th = 2.0 * np.pi * _u53(w[:, j + 1])
        out[:, j], out[:, j + 1] = r * np.cos(th), r * np.sin(th)
    return torch.from_numpy(out.reshape(-1)[:n].copy()).cuda()


def _exact_hmc(case, sigma, seed):
    d, nx, ntau, n = case["d"], case["nx"], case["ntau"], _sites(case)
    lat = _Lattice(d, nx, ntau, sigma)
    pi = _gaussian(n, 1, 0, seed).reshape(lat.shape)
    xi = torch.stack([_gaussian(n, 2, a, seed).reshape(lat.shape) for a in range(2)])
    chi = lat.MT(xi)
    for j in range(case["n_md"] + 1):
        x = lat.solve(chi)
        if j == 0:
            h0 = float(0.5 * (pi * pi).sum() + 0.5 * (chi * x).sum())
        f = -(torch.roll(lat.M(x), -1, lat.tax) * x).sum(0) * lat.sign * A_HS * torch.cos(lat.sigma)
        pi = pi - (0.5 if j in (0, case["n_md"]) else 1.0) * case["dt"] * f
        if j < case["n_md"]:
            lat = _Lattice(d, nx, ntau, lat.sigma + case["dt"] * pi)
    h1 = float(0.5 * (pi * pi).sum() + 0.5 * (chi * x).sum())
    u = float(_u53(_philox(1, 3, 0, 0, 0, seed))[0, 0])
    ok = u < math.exp(min(700.0, -(h1 - h0)))
    return {"sigma": (lat.sigma.reshape(-1) if ok else sigma.clone()), "H0": np.float64(h0),
            "H1": np.float64(h1), "accepted": int(ok)}


def _exact_observables(case, sigma, seed):
    n, k = _sites(case), case["n_noise"]
    lat = _Lattice(case["d"], case["nx"], case["ntau"], sigma, case["order"])
    eta = np.stack([np.where(_philox((n + 3) // 4, 6, j, 0, 0, seed).reshape(-1)[:n] >> np.uint64(63), 1.0, -1.0)
                    for j in range(k)])
    eta = torch.from_numpy(eta).cuda().reshape((k,) + lat.shape)
    g = eta * lat.solve(lat.MT(eta))
    t = g.reshape(k, -1).mean(1)
    ga, gb = g[:k // 2].mean(0), g[k // 2:].mean(0)
    s = torch.sin(lat.sigma)
    out = {"trace_Minv": t.mean(), "trace_err": t.std() / math.sqrt(k),
           "one_minus_g_sq": ((1.0 - ga) * (1.0 - gb)).mean(), "mean_sin": s.mean(), "mean_sin2": (s * s).mean()}
    return {name: np.float64(v.item()) for name, v in out.items()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        xs = []
        for nx, ntau, sigma, b in _batch_inputs(case, seed):
            lat = _Lattice(3, nx, ntau, torch.from_numpy(sigma).cuda())
            x = lat.solve(torch.from_numpy(b).cuda().reshape((case["n_rhs"],) + lat.shape))
            xs.append(x.reshape(b.shape).cpu().numpy())
        return {"x": xs, "failed": 0}
    inp = _inputs(case, seed)
    if kind == "hmc":
        return _exact_hmc(case, inp["sigma"], int(seed) & 0xFFFFFFFF)
    if kind == "observables":
        return _exact_observables(case, inp["sigma"], int(seed) & 0xFFFFFFFF)
    lat = _Lattice(case["d"], case["nx"], case["ntau"], inp["sigma"])
    if kind == "apply":
        return {"y": torch.stack([lat.MT(lat.M(v.double().reshape(lat.shape))).reshape(-1) for v in inp["x"]])}
    if _sites(case) * _steps(case["d"], case["ntau"]) * case["n_rhs"] > 1.2e10:
        return None          # about 20 seconds of plain CG
    b = inp["b"].reshape((case["n_rhs"],) + lat.shape)
    return {"x": lat.solve(b).reshape(case["n_rhs"], -1)}
