"""What a user of this library has it compute, as timed cases.

A case names one of the repository's workloads (``workloads``), its sizes and
one call of the public interface (``Collision``):

  eval      one sweep of C[f] and its Monte Carlo error
  euler     explicit Euler steps replayed by ``evolve``
  heun      one Heun step
  vjp, jvp  reverse- and forward-mode derivatives of the fixed-sample integral
  implicit  one backward Euler step (Newton-GMRES on jvp)

``prepare`` makes the context, the distribution and, for the derivatives, one
training sweep of the maps, as a program that differentiates has done by then.
``exact`` restates the same computation in 64-bit torch, from the published
definitions of the sample streams and the method.
"""
import math
from dataclasses import replace

import numpy as np
import torch

import workloads as W
from paper_2603_28848_gb300 import Collision

VJP_ITERATION = 0xFFFF          # Philox iteration word of the fixed-sample integral
ITEM = 8                        # samples per item of stratified sampling


# --------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------

def _case(op, problem, n, neval, nitn, precision="fp32", nbins=50, strat=False, steps=1, dt=0.1, name=None):
    c = dict(op=op, problem=problem, n=n, neval=neval, nitn=nitn, precision=precision, nbins=nbins, strat=strat,
             steps=steps, dt=dt)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a quick look while a problem is set up: few points, a ragged budget and increment count
        _case("eval", "bose", 9, 2999, 2, nbins=17, name="bose 2to2 small eval"),
        # the small Maxwell-Boltzmann run: 10 Euler steps of 5 x 1e4 samples at 32 points
        _case("euler", "mb", 32, 10_000, 5, steps=10, name="mb 2to2 euler steps"),
        # its reference-precision evaluation
        _case("eval", "mb", 32, 100_000, 2, "fp64", name="mb 2to2 fp64 eval"),
        # the flagship sweep: 128 points, two Bose species, 1e6 samples x 8
        _case("eval", "bose", 128, 1_000_000, 8, name="bose 2to2 eval"),
        # the same problem on the reference path, with the budget such checks use
        _case("eval", "bose", 128, 100_000, 2, "fp64", name="bose 2to2 fp64 eval"),
        # number-changing 2<->3 with 2->2, both pinned sides: one Heun step
        _case("heun", "cannibal", 256, 200_000, 10, dt=1e3, name="2to3 heun step"),
        # two species, three processes, expansion, m(t), budgets uneven by 100 over the grid
        _case("heun", "frw", 512, 10_000, 2, dt=0.05, name="frw multi species heun step"),
        # 2 -> 4, 12 dimensions, one sweep
        _case("eval", "fourbody", 256, 2_000_000, 2, name="2to4 eval"),
        # its gradient with respect to f, the mass and the coupling
        _case("vjp", "fourbody", 256, 400_000, 2, name="2to4 vjp"),
        # the same on the reference path, as finite-difference checks need it
        _case("vjp", "threebody", 48, 20_000, 1, "fp64", name="2to3 fp64 vjp"),
        # a stiff step: backward Euler on the 2 <-> 3 problem
        _case("implicit", "threebody", 64, 100_000, 2, dt=3e2, name="2to3 implicit step"),
        # adaptive stratified sampling (the vegas library's default mode)
        _case("eval", "bose", 128, 100_000, 5, strat=True, name="bose 2to2 stratified eval"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval2", "eval2", "eval3", "eval64", "eval64", "strat", "steps", "vjp", "jvp", "vjp64",
                       "implicit"])
    nbins = rng.choice([17, 24, 32, 50, 50, 50, 64])
    if kind == "eval2":
        c = _case("eval", rng.choice(["mb", "bose"]), _log_int(rng, 8, 160), _log_int(rng, 1e3, 1e6),
                  rng.randint(2, 8), nbins=nbins)
    elif kind == "eval3":
        c = _case("eval", rng.choice(["threebody", "cannibal", "frw", "fourbody"]), _log_int(rng, 8, 256),
                  _log_int(rng, 1e4, 2e5), 2, nbins=nbins)
    elif kind == "eval64":
        c = _case("eval", rng.choice(["mb", "bose"]), _log_int(rng, 8, 128), _log_int(rng, 5e4, 2e5),
                  rng.randint(1, 2), "fp64", nbins=nbins)
    elif kind == "strat":
        c = _case("eval", rng.choice(["mb", "bose"]), _log_int(rng, 8, 128), _log_int(rng, 1e4, 2e5),
                  rng.randint(2, 5), nbins=nbins, strat=True)
    elif kind == "steps":
        c = _case(rng.choice(["euler", "heun"]), rng.choice(["mb", "bose", "threebody"]), _log_int(rng, 8, 128),
                  _log_int(rng, 5e3, 2e5), rng.randint(2, 5), nbins=nbins, steps=rng.randint(1, 10))
    elif kind == "vjp":
        c = _case("vjp", rng.choice(["mb", "bose", "threebody", "fourbody"]), _log_int(rng, 16, 256),
                  _log_int(rng, 1e4, 4e5), 2, nbins=nbins)
    elif kind == "jvp":
        c = _case("jvp", rng.choice(["bose", "threebody", "fourbody"]), _log_int(rng, 16, 256),
                  _log_int(rng, 1e4, 4e5), 2, nbins=nbins)
    elif kind == "vjp64":
        c = _case(rng.choice(["vjp", "jvp"]), rng.choice(["mb", "bose", "threebody"]), _log_int(rng, 16, 64),
                  _log_int(rng, 5e3, 3e4), 1, "fp64", nbins=nbins)
    else:
        c = _case("implicit", "mb", _log_int(rng, 16, 64), _log_int(rng, 3e4, 2e5), 2, nbins=nbins,
                  dt=rng.uniform(3.0, 15.0))
    if c["op"] == "heun":
        c["steps"] = 1
    return c


def _problem(case, seed):
    """The workload of a case, its Philox seed and its distribution (the
    workload's own, with a smooth variation of a few percent) from `seed`."""
    n, neval, nitn = case["n"], case["neval"], case["nitn"]
    prob, f0 = {
        "mb": lambda: W.c1_maxwell_2to2(n, neval, nitn),
        "bose": lambda: W.c2_bose_2to2(n, neval, nitn),
        "threebody": lambda: W.c3_cannibal_2to3(n, neval, nitn),
        "cannibal": lambda: W.c3_cannibal_2to3(n, neval, nitn, True),
        "frw": lambda: W.c4_multi_species(n, neval, 100 * neval, nitn),
        "fourbody": lambda: W.c5_2to4(n, neval, nitn),
    }[case["problem"]]()
    procs = tuple(replace(p, nbins=case["nbins"], strat=int(case["strat"])) for p in prob.processes)
    prob = replace(prob, processes=procs, seed=prob.seed ^ (seed * 0x9E3779B97F4A7C15 & (2 ** 64 - 1)))
    rng = np.random.RandomState(seed % (2 ** 32))
    x = np.linspace(0.0, math.pi, f0.shape[1])
    wave = sum(rng.uniform(-1, 1, (f0.shape[0], 1)) * np.sin(k * x) for k in (1, 2, 3))
    return prob, f0 * np.exp(0.02 * wave)


def _time(prob):
    return 2.0 if prob.expansion is not None else 0.0


def _direction(f0, seed):
    """A cotangent / tangent direction of the size of f."""
    rng = np.random.RandomState((seed + 77) % (2 ** 32))
    return f0 * rng.uniform(-1.0, 1.0, f0.shape)


def prepare(case, seed):
    prob, f0 = _problem(case, seed)
    dev = dict(dtype=torch.float64, device="cuda")
    s = {"case": case, "t0": _time(prob)}
    s["col"] = Collision(prob, W.PREC_FP64 if case["precision"] == "fp64" else W.PREC_FP32)
    s["f"] = torch.tensor(f0, **dev)
    if case["op"] in ("vjp", "jvp"):
        s["dir"] = torch.tensor(_direction(f0, seed), **dev)
        s["col"].eval(s["f"], s["t0"])
    if case["op"] in ("euler", "heun", "implicit"):
        s["logf0"] = torch.log(s["f"])
        s["logf"] = s["logf0"].clone()
        s["t"] = torch.tensor([s["t0"]], **dev)
        s["dt"] = torch.tensor([case["dt"]], **dev)
    return s


def run(s):
    case, col = s["case"], s["col"]
    op = case["op"]
    if op == "eval":
        return col.eval(s["f"], s["t0"])
    if op == "vjp":
        return col.vjp(s["f"], s["dir"], s["t0"])
    if op == "jvp":
        return col.jvp(s["f"], s["dir"], s["t0"])
    s["logf"].copy_(s["logf0"])
    if op == "implicit":
        col.step_implicit_euler(s["logf"], s["t0"], case["dt"])
        return s["logf"]
    s["t"].fill_(s["t0"])
    s["dt"].fill_(case["dt"])
    if op == "euler":
        col.evolve(s["logf"], s["t"], s["dt"], case["steps"], case["dt"], "euler")
    else:
        col.step_heun(s["logf"], s["t"], s["dt"])
    return s["logf"], s["t"]


# --------------------------------------------------------------------------
# the work of one pass
# --------------------------------------------------------------------------

def _sides(prob):
    """Side integrals of Eq. (7): process, side, observed species and leg,
    multiplicity, conserved leg and integrated legs of App. A."""
    out = []
    for pi, p in enumerate(prob.processes):
        n_in, legs = len(p.species_in), tuple(p.species_in) + tuple(p.species_out)
        n = len(legs)
        same = sorted(p.species_in) == sorted(p.species_out)
        for side in range(1 if same else 2):
            own = range(n_in) if side == 0 else range(n_in, n)
            for sp in sorted({legs[k] for k in own}):
                mine = [k for k in own if legs[k] == sp]
                obs = mine[0]
                if n_in != n - n_in:
                    first = range(n_in) if n_in < n - n_in else range(n_in, n)
                else:
                    first = own
                order = list(first) + [k for k in range(n) if k not in first]
                cons = next(k for k in order if k != obs)
                out.append(dict(process=pi, p=p, legs=legs, n_in=n_in, own=set(own), species=sp, obs=obs,
                                mult=len(mine), cons=cons, integ=[k for k in range(n) if k not in (obs, cons)]))
    return out


def _budgets(prob, side):
    p = side["p"]
    N = np.full(prob.grid.n, p.neval) if p.neval_per_point is None else np.array(p.neval_per_point)
    return N // ITEM * ITEM if p.strat else N


def _samples(prob):
    """(samples, samples x integrated legs) of one VEGAS iteration of every task."""
    tot = legs = 0
    for s in _sides(prob):
        k = 2 * int(_budgets(prob, s).sum())
        tot += k
        legs += k * len(s["integ"])
    return tot, legs


def _passes(case):
    """Iterations of every sample that one pass draws."""
    return {"eval": case["nitn"], "euler": case["nitn"] * case["steps"], "heun": 2 * case["nitn"], "vjp": 1, "jvp": 1,
            "implicit": case["nitn"] + 8}[case["op"]]


def work(case):
    prob, f0 = _problem(case, 1)
    tot, legs = _samples(prob)
    # per sample 48 operations for each integrated leg and 40 for the rest (FMA = 2); the reverse and
    # forward derivatives of one sample cost about as much again
    flops = _passes(case) * (48.0 * legs + 40.0 * tot) * (2.0 if case["op"] in ("vjp", "jvp") else 1.0)
    if case["op"] == "implicit":
        flops = (case["nitn"] + 2.0 * 8) * (48.0 * legs + 40.0 * tot)
    maps = 2 * prob.grid.n * sum(3 * len(s["integ"]) * (s["p"].nbins + 1) for s in _sides(prob)) * 8
    return {"bytes": float(maps * (1 if case["op"] in ("vjp", "jvp") else 2) + 6 * f0.size * 8), "flops": flops}


# --------------------------------------------------------------------------
# the same in 64-bit torch
# --------------------------------------------------------------------------

M32 = 0xFFFFFFFF


def _philox(block, itn, call, task, seed):
    """Philox4x32-10 words (int64 tensors of 32-bit values), shape block.shape + (4,)."""
    c0 = block & M32
    c1, c2, c3 = (torch.full_like(c0, itn), torch.full_like(c0, call), task.expand_as(c0))
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57          # mod 2^64 in two's complement
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return torch.stack((c0, c1, c2, c3), -1)


class _Exact:
    """The method in 64 bits: maps, stratified allocations and the evaluation
    counter of one context."""

    def __init__(self, prob, f32):
        self.prob, self.f32 = prob, f32
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        g = prob.grid
        q = g.q_min * (g.q_max / g.q_min) ** (np.arange(g.n) / (g.n - 1))
        q[0], q[-1] = g.q_min, g.q_max
        self.q = torch.tensor(q, device=self.dev)
        self.call = 0
        self.sides = _sides(prob)
        for s in self.sides:
            s["D"] = 3 * len(s["integ"])
            nb = s["p"].nbins
            s["map"] = (torch.arange(nb + 1, device=self.dev, dtype=torch.float64) / nb).repeat(2 * g.n, s["D"], 1)
            s["N"] = torch.tensor(np.repeat(_budgets(prob, s), 2), device=self.dev)
            if s["p"].strat:
                J, D = s["p"].neval // ITEM, s["D"]
                M = 1
                while 4 * (M + 1) ** D <= J and (M + 1) ** D <= s["p"].strat_max_hcubes:
                    M += 1
                H = M ** D
                m = torch.full((2 * g.n, H), J // H, device=self.dev, dtype=torch.int64)
                m[:, : J % H] += 1
                s["strat"] = (M, H, J, m)
        self.lam = torch.tensor([p.coupling for p in prob.processes], dtype=torch.float64, device=self.dev)

    def masses(self, t):
        return torch.tensor([s.mass0 + s.mass1 * t for s in self.prob.species], dtype=torch.float64, device=self.dev)

    def begin(self, f, t, m=None, lam=None):
        """Splines and tails of f (differentiable) at time t."""
        ex, q, n = self.prob.expansion, self.q, self.prob.grid.n
        self.a = 1.0 if ex is None else ex.a0 * math.sqrt(t / ex.t0)
        self.m = self.masses(t) if m is None else m
        self.lam_now = self.lam if lam is None else lam
        self.f = f
        self.eta = [(0.0, 1.0, -1.0)[s.stat] for s in self.prob.species]
        h = q[1:] - q[:-1]
        A = torch.zeros(n, n, dtype=torch.float64, device=self.dev)      # not-a-knot system of the second derivatives
        i = torch.arange(1, n - 1, device=self.dev)
        A[i, i - 1], A[i, i], A[i, i + 1] = h[:-1], 2 * (h[:-1] + h[1:]), h[1:]
        A[0, :3] = torch.stack((h[1], -(h[0] + h[1]), h[0]))
        A[-1, -3:] = torch.stack((h[-1], -(h[-1] + h[-2]), h[-2]))
        d = (f[:, 1:] - f[:, :-1]) / h
        zero = torch.zeros_like(f[:, :1])
        rhs = torch.cat((zero, 6 * (d[:, 1:] - d[:, :-1]), zero), 1)
        s2 = rhs @ torch.linalg.inv(A).T
        self.coef = torch.stack((f[:, :-1], d - h * (2 * s2[:, :-1] + s2[:, 1:]) / 6, s2[:, :-1] / 2,
                                 (s2[:, 1:] - s2[:, :-1]) / (6 * h)), -1)
        self.tail = []
        K = self.prob.tail_points
        for sp, eta in enumerate(self.eta):
            ends = []
            for sl in (slice(0, K), slice(n - K, n)):
                x = torch.sqrt((q[sl] / self.a) ** 2 + self.m[sp] ** 2)
                y = torch.log(1 / f[sp, sl] + eta)
                xc = x - x.mean()
                b = (xc * (y - y.mean())).sum() / (xc * xc).sum()
                ends.append((y.mean() - b * x.mean(), b))
            self.tail.append(ends)

    def lookup(self, sp, r):
        j = torch.searchsorted(self.q, r.detach(), right=True).sub_(1).clamp_(0, self.prob.grid.n - 2)
        x = r - self.q[j]
        c = self.coef[sp][j]
        v = ((c[..., 3] * x + c[..., 2]) * x + c[..., 1]) * x + c[..., 0]
        v = torch.where(v > 0, v, torch.zeros_like(v))
        return torch.where(v < 1, v, torch.ones_like(v)) if self.eta[sp] < 0 else v

    def draw(self, s, tasks, s0, s1, itn):
        """Increments [T, S, D] and fractions of samples s0 .. s1 of the tasks (s0 a multiple of 4)."""
        D, per = s["D"], 4 if self.f32 else 2
        b0, b1 = s0 * D // per, -(-s1 * D // per)
        block = torch.arange(b0, b1, device=self.dev).expand(len(tasks), -1)
        gid = self.sides.index(s) * 2 * self.prob.grid.n + tasks
        w = _philox(block, itn, self.call, gid[:, None], self.prob.seed)
        if self.f32:
            u = w.double() * 2.0 ** -32
        else:
            k = ((w[..., 0::2] >> 6) << 26) | (w[..., 1::2] >> 6)
            u = (k.double() + 0.5) * 2.0 ** -52
        u = u.reshape(len(tasks), -1)[:, : (s1 - s0) * D].reshape(len(tasks), s1 - s0, D)
        h = None
        if s["p"].strat:
            M, H, J, m = s["strat"]
            item = torch.arange(s0, s1, device=self.dev) // ITEM
            h = torch.searchsorted(m[tasks].cumsum(1), item.expand(len(tasks), -1).contiguous(), right=True).clamp_(max=H - 1)
            u = (torch.stack([h // M ** d % M for d in range(D)], -1) + u) / M
        nb = s["p"].nbins
        x = u * nb
        b = x.floor().clamp_(max=nb - 1).long()
        return b, x - b, h

    def weights(self, s, tasks, b, fr):
        """Sample weights w [T, S] of Eq. (12)."""
        p, a, nb = s["p"], self.a, s["p"].nbins
        g = self.prob.grid
        T, S, D = b.shape
        e = s["map"][tasks]
        flat = b.transpose(1, 2)
        lo = torch.gather(e, 2, flat.reshape(T, D, S))
        dy = torch.gather(e, 2, flat.reshape(T, D, S) + 1) - lo
        y = lo + fr.transpose(1, 2) * dy
        jac = (dy * nb).prod(1)
        point, loss = tasks // 2, (tasks % 2 == 1)[:, None]
        p_obs = (self.q[point] / a)[:, None]
        m_obs = self.m[s["species"]]
        E_obs = torch.sqrt(p_obs ** 2 + m_obs ** 2)
        sign = lambda k: 1.0 if k < s["n_in"] else -1.0
        f_obs = self.f[s["species"]][point][:, None]
        w = torch.where(loss, f_obs, 1 + self.eta[s["species"]] * f_obs)
        balance = sign(s["obs"]) * E_obs
        px = py = 0.0
        pz = sign(s["obs"]) * p_obs
        keep = E_obs >= self.prob.e_cut

        def factor(w, k, f):
            eta = self.eta[s["legs"][k]]
            enhanced = (k in s["own"]) != loss
            return w * torch.where(enhanced, 1 + eta * f, f)

        for i, k in enumerate(s["integ"]):
            r = g.q_min + (g.q_max - g.q_min) * y[:, 3 * i]
            th, ph = math.pi * y[:, 3 * i + 1], 2 * math.pi * y[:, 3 * i + 2]
            st, pk = torch.sin(th), r / a
            px, py, pz = (px + sign(k) * pk * st * torch.cos(ph), py + sign(k) * pk * st * torch.sin(ph),
                          pz + sign(k) * pk * torch.cos(th))
            E = torch.sqrt(pk ** 2 + self.m[s["legs"][k]] ** 2)
            keep = keep & (E >= self.prob.e_cut)
            balance = balance + sign(k) * E
            jac = jac * (g.q_max - g.q_min) * 2 * math.pi ** 2 * r * r * st / E
            w = factor(w, k, self.lookup(s["legs"][k], r))
        k = s["cons"]
        sp = s["legs"][k]
        pc = torch.sqrt(px * px + py * py + pz * pz)
        E = torch.sqrt(pc ** 2 + self.m[sp] ** 2)
        keep = keep & (E >= self.prob.e_cut)
        balance = balance + sign(k) * E
        qc = pc * a
        fc = self.lookup(sp, qc.clamp(g.q_min, g.q_max))
        for (ta, tb), out in zip(self.tail[sp], (qc < g.q_min, qc > g.q_max)):
            x = torch.where(out, ta + tb * E, torch.ones_like(E))
            den = torch.expm1(x) if self.eta[sp] > 0 else torch.exp(x) - self.eta[sp]
            ft = torch.where(den > 0, 1 / torch.where(den > 0, den, torch.ones_like(den)), torch.zeros_like(den))
            if self.eta[sp] < 0:
                ft = torch.where(ft < 1, ft, torch.ones_like(ft))
            fc = torch.where(out, ft, fc)
        w = factor(w, k, fc)
        n = len(s["legs"])
        sig = p.sigma_E
        K = self.lam_now[s["process"]] ** 2 * a ** (-3 * (n - 2)) / (
            (2 * math.pi) ** (3 * (n - 1) - 4) * 2.0 ** n * E_obs * sig * math.sqrt(2 * math.pi))
        w = w * K * jac / E * torch.exp(-balance ** 2 / (2 * sig * sig))
        return torch.where(keep, w, torch.zeros_like(w))

    def batches(self, s, limit):
        """Groups of tasks of similar budgets and ranges of their samples, of at most `limit` sample dimensions."""
        order = torch.argsort(s["N"], descending=True, stable=True).cpu().numpy()
        N = s["N"].cpu().numpy()
        k = 0
        while k < len(order):
            top = int(N[order[k]])
            room = max(1, limit // (top * s["D"]))
            j = k
            while j < len(order) and j - k < room and N[order[j]] * 1.25 >= top:
                j += 1
            step = max(ITEM, limit // ((j - k) * s["D"]) // ITEM * ITEM)
            yield torch.tensor(order[k:j], device=self.dev), [(x, min(top, x + step)) for x in range(0, top, step)]
            k = j

    def refine(self, s, tasks, hist):
        nb = s["p"].nbins
        d = torch.cat((hist[..., :1], hist, hist[..., -1:]), -1)
        d = (d[..., :-2] + 6 * d[..., 1:-1] + d[..., 2:]) / 8
        tot = d.sum(-1, keepdim=True)
        v = d / torch.where(tot > 0, tot, torch.ones_like(tot))
        inside = (v >= 1e-30) & (v < 1)
        vi = torch.where(inside, v, torch.full_like(v, 0.5))
        o = torch.where(inside, ((1 - vi) / -torch.log(vi)) ** s["p"].alpha, (v >= 1).double())
        cum = torch.cat((torch.zeros_like(tot), o.cumsum(-1)), -1)
        goal = cum[..., -1:] / nb * torch.arange(1, nb, device=self.dev)
        i = torch.searchsorted(cum[..., 1:].contiguous(), goal.contiguous()).clamp_(max=nb - 1)
        fr = ((goal - cum.gather(-1, i)) / o.gather(-1, i)).clamp(0, 1)
        old = s["map"][tasks]
        lo, hi = old.gather(-1, i), old.gather(-1, i + 1)
        new = old.clone()
        new[..., 1:-1] = lo + fr * (hi - lo)
        s["map"][tasks] = torch.where(tot > 0, new, old)

    def sweep(self, f, t):
        """C and its error of one evaluation; refines the maps."""
        self.begin(f, t)
        C, var = torch.zeros_like(f), torch.zeros_like(f)
        for s in self.sides:
            nb, D = s["p"].nbins, s["D"]
            mean, err2 = (torch.zeros(2 * self.prob.grid.n, dtype=torch.float64, device=self.dev) for _ in range(2))
            for tasks, ranges in self.batches(s, 24_000_000):
                T = len(tasks)
                N = s["N"][tasks].double()
                inv, minv = torch.zeros(T, device=self.dev).double(), torch.zeros(T, device=self.dev).double()
                exact, n_exact = inv.clone(), inv.clone()
                for itn in range(s["p"].nitn):
                    s1, s2 = torch.zeros(T, device=self.dev).double(), torch.zeros(T, device=self.dev).double()
                    hist = torch.zeros(T * D * nb, dtype=torch.float64, device=self.dev)
                    if s["p"].strat:
                        M, H, J, m_all = s["strat"]
                        m = m_all[tasks].double()
                        h1, h2 = torch.zeros(2, T, H, dtype=torch.float64, device=self.dev)
                    for x0, x1 in ranges:
                        b, fr, h = self.draw(s, tasks, x0, x1, itn)
                        w = self.weights(s, tasks, b, fr)
                        w = torch.where(torch.arange(x0, x1, device=self.dev) < N[:, None], w, torch.zeros_like(w))
                        w2 = w * w
                        s1 += w.sum(1)
                        s2 += w2.sum(1)
                        if h is not None:
                            h1.scatter_add_(1, h, w)
                            h2.scatter_add_(1, h, w2)
                            w2 = w2 / m.gather(1, h)
                        row = (torch.arange(T, device=self.dev)[:, None] * D + torch.arange(D, device=self.dev)) * nb
                        for d in range(D):
                            hist.index_add_(0, (row[:, d, None] + b[..., d]).reshape(-1), w2.reshape(-1))
                    if s["p"].strat:
                        n = ITEM * m
                        v2 = ((h2 - h1 * h1 / n) / (n - 1)).clamp(min=0)
                        mu, v = (h1 / n).sum(1) / H, (v2 / n).sum(1) / H ** 2
                        share = v2 ** (0.5 * s["p"].strat_beta)
                        tot = share.sum(1, keepdim=True)
                        new = 1 + torch.floor((J - H) * share / tot).long()
                        new += (torch.arange(H, device=self.dev) < (J - new.sum(1, keepdim=True))).long()
                        m_all[tasks] = torch.where(tot > 0, new, m_all[tasks])
                    else:
                        mu = s1 / N
                        v = ((s2 / N - mu * mu) / (N - 1)).clamp(min=0)
                    ok = v > 0
                    vi = torch.where(ok, v, torch.ones_like(v))
                    inv += torch.where(ok, 1 / vi, torch.zeros_like(v))
                    minv += torch.where(ok, mu / vi, torch.zeros_like(v))
                    exact += torch.where(ok, torch.zeros_like(v), mu)
                    n_exact += (~ok).double()
                    self.refine(s, tasks, hist.reshape(T, D, nb))
                some = n_exact > 0
                one = torch.ones_like(inv)
                iv = torch.where(inv > 0, inv, one)
                mean[tasks] = torch.where(some, exact / torch.where(some, n_exact, one), minv / iv)
                err2[tasks] = torch.where(some, torch.zeros_like(inv), torch.where(inv > 0, 1 / iv, torch.zeros_like(inv)))
            C[s["species"]] += s["mult"] * (mean[0::2] - mean[1::2])
            var[s["species"]] += s["mult"] ** 2 * (err2[0::2] + err2[1::2])
        self.call += 1
        return C, torch.sqrt(var)

    def fixed(self, f, t, u=None):
        """C~ of the fixed-sample integral and, with u, its tangent along u."""
        import torch.autograd.forward_ad as fwd
        C, JU = torch.zeros_like(f), torch.zeros_like(f)
        for s in self.sides:
            for tasks, ranges in self.batches(s, 12_000_000):
                N = s["N"][tasks].double()
                for x0, x1 in ranges:
                    b, fr, _ = self.draw(s, tasks, x0, x1, VJP_ITERATION)
                    with fwd.dual_level():
                        self.begin(f if u is None else fwd.make_dual(f, u), t)
                        w = self.weights(s, tasks, b, fr)
                        w = torch.where(torch.arange(x0, x1, device=self.dev) < N[:, None], w, torch.zeros_like(w))
                        val, tan = fwd.unpack_dual(s["mult"] * w.sum(1) / N * (1 - 2 * (tasks % 2)))
                    C[s["species"]].index_add_(0, tasks // 2, val)
                    if u is not None:
                        JU[s["species"]].index_add_(0, tasks // 2, tan)
        return C, JU

    def gradients(self, f, t, v=None):
        """C~ and the gradients of sum(v C~) by f, the masses and the couplings;
        without v the rows dC~_a(p_i)/df instead, [S n, S n]."""
        C = torch.zeros_like(f)
        leaf = [x.clone().requires_grad_(True) for x in (f, self.masses(t), self.lam)]
        rows = torch.zeros(f.numel(), f.numel(), dtype=torch.float64, device=self.dev) if v is None else None
        n = self.prob.grid.n
        for s in self.sides:
            groups = self.batches(s, 3_000_000) if v is not None else (
                (torch.tensor([2 * i, 2 * i + 1], device=self.dev), [(0, int(s["N"][2 * i]))]) for i in range(n))
            for tasks, ranges in groups:
                N = s["N"][tasks].double()
                for x0, x1 in ranges:
                    b, fr, _ = self.draw(s, tasks, x0, x1, VJP_ITERATION)
                    self.begin(leaf[0], t, leaf[1], leaf[2])
                    w = self.weights(s, tasks, b, fr)
                    w = torch.where(torch.arange(x0, x1, device=self.dev) < N[:, None], w, torch.zeros_like(w))
                    I = s["mult"] * w.sum(1) / N * (1 - 2 * (tasks % 2))
                    C[s["species"]].index_add_(0, tasks // 2, I.detach())
                    if v is not None:
                        (I * v[s["species"]][tasks // 2]).sum().backward()
                    else:
                        (gf,) = torch.autograd.grad(I.sum(), leaf[0])
                        rows[s["species"] * n + int(tasks[0]) // 2] += gf.reshape(-1)
        return (C, *(x.grad for x in leaf)) if v is not None else (C, rows)

    def implicit(self, logf, t, dt):
        """Backward Euler of log f by Newton's method (dense Jacobian, halved steps), after one training sweep."""
        self.sweep(torch.exp(logf), t + dt)

        def residual(x):
            f = torch.exp(x)
            return x - logf - dt * self.fixed(f, t + dt)[0] / f

        x, res = logf.clone(), residual(logf)
        for _ in range(12):
            if float(res.abs().max()) < 1e-9:
                break
            f = torch.exp(x)
            C, J = self.gradients(f, t + dt)
            fv, Cv = f.reshape(-1), C.reshape(-1)
            A = torch.diag(1 + dt * Cv / fv) - dt * J * (fv / fv[:, None])
            d = torch.linalg.solve(A, res.reshape(-1)).reshape(x.shape)
            for half in range(12):
                trial = x - d * 0.5 ** half
                new = residual(trial)
                if float(new.norm()) < float(res.norm()):
                    break
            x, res = trial, new
        return x


def _settled(case):
    """Whether 64-bit arithmetic on the same samples determines what FP32 returns beyond its rounding: training
    data in FP32 move the next iteration's samples, and after several iterations (or reallocations, or in many
    dimensions) these are other samples of the same integral."""
    if case["precision"] == "fp64" or case["op"] == "implicit":
        return True
    two = case["problem"] in ("mb", "bose")
    if case["strat"] or (case["op"] in ("eval", "vjp", "jvp") and not two):
        return False
    return case["op"] != "eval" or case["nitn"] <= 2 or case["neval"] >= 500_000


def exact(case, seed):
    prob, f0 = _problem(case, seed)
    tot, legs = _samples(prob)
    # sample dimensions x passes over them, weighted by what a derivative costs
    cost = 3 * legs * {"vjp": 24, "jvp": 4, "implicit": case["nitn"] + 120}.get(case["op"], _passes(case))
    if cost > 3e10 or not _settled(case):
        return None
    ex = _Exact(prob, case["precision"] == "fp32")
    t = _time(prob)
    f = torch.tensor(f0, device=ex.dev)
    op = case["op"]
    if op == "eval":
        return ex.sweep(f, t)
    if op in ("vjp", "jvp"):
        d = torch.tensor(_direction(f0, seed), device=ex.dev)
        ex.sweep(f, t)
        return ex.gradients(f, t, d) if op == "vjp" else ex.fixed(f, t, d)
    logf = torch.log(f)
    if op == "implicit":
        return ex.implicit(logf, t, case["dt"])
    dt = case["dt"]
    for _ in range(case["steps"]):
        f = torch.exp(logf)
        k1, _ = ex.sweep(f, t)
        top = float((k1 / f).abs().max())
        step = min(case["dt"], prob.eps_dt / top) if top > 0 else case["dt"]
        if op == "euler":
            logf = logf + step * k1 / f
        else:
            fs = torch.exp(logf + step * k1 / f)
            k2, _ = ex.sweep(fs, t + step)
            logf = logf + 0.5 * step * (k1 / f + k2 / fs)
        t = t + step
    # the step taken follows the largest C/f, of one noisy point: in FP32 not settled by these samples
    return logf, (torch.tensor([t], dtype=torch.float64, device=ex.dev) if case["precision"] == "fp64" else None)
