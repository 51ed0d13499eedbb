"""The workloads this framework is timed on: single-chain updates, proposals and
moments, and batches of chains, through the public Python binding.

A case is one call a user's program repeats: ``updates`` (a block of Metropolis
updates of one chain, Algorithm 1), ``delta_omega`` (one proposal evaluated),
``moments`` (the 7x7 local moments of one site), ``batch`` (one launch over many
chains on teams of CTAs) and ``plan`` (one captured step of a batch, on teams or
on thread-block clusters).  Sizes are those of the tests, the benchmark and the
serving and temperature-scan modules: L = 4 .. 48, M = 256 .. 2048, FP64 and
FP32-mixed, both recursions, t = 1, a = 6.05.

FP32-mixed chains give Delta Omega with the accuracy of their FP32 vectors, so
those traces are returned as float32; FP64 chains return float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1303_6016_gb300 import batch, gfmc, inputs

SCALE = 6.05  # spectral scale a (t = 1)


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _chain(name, call, L, M, n, precision="fp64", recursion="unit_vectors", spins="uniform", kernel="jackson",
           nodes=0, beta=20.0, mu=-2.0):
    return {"name": name, "call": call, "L": L, "M": M, "updates": n, "precision": precision,
            "recursion": recursion, "spins": spins, "kernel": kernel, "nodes": nodes, "beta": beta, "mu": mu}


def _many(name, call, schedule, sizes, chains, M, n, precision="fp32_mixed", recursion="unit_vectors",
          spins="uniform", tmin=0.02, tmax=0.2, mu=-2.0):
    return {"name": name, "call": call, "schedule": schedule, "sizes": sizes, "chains": chains, "M": M,
            "updates": n, "precision": precision, "recursion": recursion, "spins": spins, "tmin": tmin,
            "tmax": tmax, "mu": mu}


def listed():
    return [
        # a program that evaluates single proposals (a custom update rule, a check): the smallest call
        _chain("delta_omega_L6", "delta_omega", 6, 256, 1),
        # one sequential sweep of the smallest lattice of the paper's validation
        _chain("sweep_L4", "updates", 4, 256, 64),
        # inspecting the local moments (local density of states) of a site
        _chain("moments_L12", "moments", 12, 512, 1),
        # an odd lattice (no parity split), Lorentz kernel, 2M nodes
        _chain("updates_L9_odd", "updates", 9, 512, 16, spins="vmf", kernel="lorentz", nodes=1024),
        # single FP64 chains: the medium lattice, and the headline workload
        _chain("updates_L16", "updates", 16, 1024, 16),
        _chain("updates_L32", "updates", 32, 1024, 16),
        # the headline workload in FP32-mixed
        _chain("updates_L32_fp32", "updates", 32, 1024, 32, precision="fp32_mixed"),
        # the headline workload on the proposal's vectors
        _chain("updates_L32_proposal", "updates", 32, 1024, 16, recursion="proposal"),
        # the largest lattice of the serving mix, as its jobs run it
        _chain("updates_L48_proposal", "updates", 48, 512, 4, recursion="proposal", spins="vmf"),
        # the temperature scan: many small chains, one CTA each, mu = 0
        _many("scan_L4_8", "batch", "ones", "4,6,8", 24, 256, 64, spins="vmf", tmin=0.02, tmax=0.3, mu=0.0),
        # 64 chains of mixed sizes, captured steps: teams of CTAs, and clusters
        _many("plan_teams", "plan", "teams", "8,12,16,24,32", 64, 1024, 2),
        _many("plan_clusters", "plan", "clusters", "8,12,16,24,32", 64, 1024, 4, recursion="proposal"),
    ]


def draw(rng):
    M = rng.choice([256, 512, 1024, 1024, 2048])
    spins = rng.choice(["uniform", "vmf"])
    precision = rng.choice(["fp64", "fp32_mixed"])
    kind = rng.choice(["updates"] * 5 + ["delta_omega", "moments", "batch", "plan", "plan"])
    if kind in ("batch", "plan"):
        M = min(M, 1024)
        chains = rng.randint(8, 64)
        top = rng.choice([8, 12, 16, 24, 32]) if kind == "plan" else 8
        sizes = sorted(rng.sample([s for s in (4, 5, 6, 8, 10, 12, 16, 20, 24, 32) if s <= top], 3))
        schedule = "ones" if kind == "batch" else rng.choice(["teams", "clusters"])
        recursion = "proposal" if schedule == "clusters" else rng.choice(["unit_vectors", "proposal"])
        n = rng.randint(8, 32) if kind == "batch" else rng.randint(1, 2)
        return {"call": kind, "schedule": schedule, "sizes": ",".join(map(str, sizes)), "chains": chains, "M": M,
                "updates": n, "precision": "fp32_mixed", "recursion": recursion, "spins": spins, "tmin": 0.02,
                "tmax": 0.2, "mu": rng.choice([-2.0, 0.0])}
    L = int(round(math.exp(rng.uniform(math.log(4), math.log(40)))))
    if L % 2 and rng.random() < 0.5:
        L += 1  # even lattices are the usual choice
    budget = 2.0 ** 27 * (4 if precision == "fp32_mixed" else 1)
    n = 1
    if kind == "updates":
        n = max(1, min(rng.randint(2, 64), int(budget / (float(L) ** 3 * M)), 20000 // M))
    return {"call": kind, "L": L, "M": M, "updates": n, "precision": precision,
            "recursion": rng.choice(["unit_vectors", "unit_vectors", "proposal"]), "spins": spins,
            "kernel": rng.choice(["jackson", "jackson", "jackson", "lorentz"]),
            "nodes": 2 * M if rng.random() < 0.2 else 0, "beta": rng.choice([5.0, 10.0, 20.0, 50.0]),
            "mu": rng.choice([-2.0, 0.0])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _spins(case, L, seed):
    return inputs.von_mises_fisher(L, 5.0, seed) if case["spins"] == "vmf" else inputs.uniform_sphere(L, seed)


def _members(case, seed):
    """Lattice size, inverse temperature and spins of each chain of a batch."""
    rng = np.random.default_rng(seed)
    sizes = [int(s) for s in case["sizes"].split(",")]
    # every size equally often, as near as it goes, so that another seed is the same work
    Ls = sorted(sizes[c % len(sizes)] for c in range(case["chains"]))
    betas = 1.0 / rng.uniform(case["tmin"], case["tmax"], size=len(Ls))
    return Ls, betas, [_spins(case, L, 1000 * (seed % 100000) + c) for c, L in enumerate(Ls)]


def _teams(Ls, budget):
    """CTAs per chain: one each, the rest to the chains with the most sites per CTA."""
    t = [1] * len(Ls)
    for _ in range(budget - len(Ls)):
        c = max(range(len(Ls)), key=lambda q: Ls[q] ** 3 / t[q])
        if t[c] >= 32 or Ls[c] ** 3 / t[c] <= 512:
            break
        t[c] += 1
    return t


def _probe(case, seed):
    """Site and proposed direction of a single evaluation."""
    rng = np.random.default_rng(seed + 77)
    return int(rng.integers(case["L"] ** 3)), float(np.arccos(1 - 2 * rng.random())), float(2 * np.pi * rng.random())


def prepare(case, seed):
    if case["call"] in ("batch", "plan"):
        Ls, betas, spins = _members(case, seed)
        chains = [gfmc.Chain(L, s, M=case["M"], beta=float(b), mu=case["mu"], precision=case["precision"],
                             seed=1 + seed, chain_id=c, recursion=case["recursion"])
                  for c, (L, b, s) in enumerate(zip(Ls, betas, spins))]
        state = {"case": case, "chains": chains}
        if case["schedule"] == "clusters":
            ctas = [gfmc.cluster_min_ctas(L, case["M"], case["precision"]) for L in Ls]
        elif case["schedule"] == "teams":
            ctas = _teams(Ls, batch.device_ctas())
        else:
            ctas = [1] * len(Ls)
        state["ctas"] = ctas
        if case["call"] == "plan":
            # the largest chains first, as the batch runners issue them
            order = sorted(range(len(Ls)), key=lambda c: -Ls[c])
            state["plan"] = gfmc.Plan([chains[c] for c in order], case["updates"], [ctas[c] for c in order],
                                      schedule=case["schedule"])
        return state
    ch = gfmc.Chain(case["L"], _spins(case, case["L"], seed), M=case["M"], beta=case["beta"], mu=case["mu"],
                    precision=case["precision"], kernel=case["kernel"], seed=1 + seed, recursion=case["recursion"],
                    nodes=case["nodes"])
    return {"case": case, "chain": ch, "probe": _probe(case, seed)}


def _real(case, x):
    return np.asarray(x, dtype=np.float32 if case["precision"] == "fp32_mixed" else np.float64)


def run(state):
    case = state["case"]
    if case["call"] == "moments":
        mu = state["chain"].moments(state["probe"][0])
        return mu.astype(np.complex64) if case["precision"] == "fp32_mixed" else mu
    if case["call"] == "delta_omega":
        return _real(case, [state["chain"].delta_omega(*state["probe"])])
    if case["call"] == "updates":
        out = state["chain"].updates(case["updates"])
        return {"d_omega": _real(case, out["d_omega"]), "decisions": out["decisions"],
                "spins": state["chain"].get_spins()}
    if case["call"] == "batch":
        res = gfmc.run_batch(state["chains"], case["updates"], team_ctas=state["ctas"])
    else:
        state["plan"].launch(1)
        res = state["plan"].sync()
    return {"d_omega": _real(case, np.concatenate([r["d_omega"] for r in res])),
            "decisions": np.concatenate([r["decisions"] for r in res]),
            "n_accepted": np.array([r["n_accepted"] for r in res])}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def work(case):
    """Delta Omega needs <o|T_n|o>, <v|T_n|v> and <o|T_n|v>: M/2 steps of two
    vectors and their products (56 flop per site on an even lattice, where each
    vector lives on one parity); moments need all seven vectors and the products
    of the 7x7 blocks (280 flop per site on an even lattice).  Bytes: the spins
    read and the results written."""
    def flops(L, M, vectors7):
        per = (280 if L % 2 == 0 else 791) if vectors7 else (56 if L % 2 == 0 else 128)
        return (M // 2 - 1) * L ** 3 * per

    if case["call"] in ("batch", "plan"):
        sizes = [int(s) for s in case["sizes"].split(",")]
        Ls = [sizes[c % len(sizes)] for c in range(case["chains"])]
        return {"bytes": sum(16 * L ** 3 + 9 * case["updates"] for L in Ls),
                "flops": case["updates"] * sum(flops(L, case["M"], False) for L in Ls)}
    L, M, n = case["L"], case["M"], case["updates"]
    out = 49 * M * 16 if case["call"] == "moments" else 9 * n
    spins = 2 if case["call"] == "updates" else 1
    return {"bytes": spins * 16 * L ** 3 + out, "flops": n * flops(L, M, case["call"] == "moments")}


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ---------------------------------------------------------------------------
def _philox(key0, key1, ctr):
    """Philox4x32-10 (Salmon et al., SC'11) of the counter (ctr, 0, 0, 0)."""
    m32 = 0xFFFFFFFF
    c, k = [ctr & m32, ctr >> 32, 0, 0], [key0 & m32, key1 & m32]
    for r in range(10):
        if r:
            k = [(k[0] + 0x9E3779B9) & m32, (k[1] + 0xBB67AE85) & m32]
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [(p1 >> 32) ^ c[1] ^ k[0], p1 & m32, (p0 >> 32) ^ c[3] ^ k[1], p0 & m32]
    return c


class _Exact:
    """B chains of one lattice size, advanced together by the plain Chebyshev
    recursion (no doubling, no FFT), in complex128."""

    def __init__(self, L, spins, M, beta, mu, kernel="jackson", K=0):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.L, self.N, self.M, self.K = L, L ** 3, M, K or M
        self.spins = torch.tensor(np.asarray(spins), device=self.dev)  # [B, N, 2]
        self.B = self.spins.shape[0]
        i = np.arange(self.N)
        x, y, z = i % L, (i // L) % L, i // (L * L)
        nb = [(x + 1) % L + L * (y + L * z), (x - 1) % L + L * (y + L * z), x + L * ((y + 1) % L + L * z),
              x + L * ((y - 1) % L + L * z), x + L * (y + L * ((z + 1) % L)), x + L * (y + L * ((z - 1) % L))]
        self.nb = torch.tensor(np.stack(nb), device=self.dev)
        n = torch.arange(M, device=self.dev, dtype=torch.float64)
        if kernel == "jackson":
            q = math.pi / (M + 1)
            g = ((M - n + 1) * torch.cos(q * n) + torch.sin(q * n) / math.tan(q)) / (M + 1)
        else:
            g = torch.sinh(4.0 * (1 - n / M)) / math.sinh(4.0)
        th = math.pi * (torch.arange(self.K, device=self.dev, dtype=torch.float64) + 0.5) / self.K
        self.sin = torch.sin(th)
        # G(w_k) = (i / sin theta_k) [g_0 mu_0 + 2 sum_n g_n mu_n e^{-i n theta_k}]
        ph = torch.outer(th, n)
        self.green = torch.complex(torch.cos(ph), -torch.sin(ph)) * (g * torch.where(n > 0, 2.0, 1.0))
        self.green = self.green * (1j / self.sin)[:, None]
        E = SCALE * torch.cos(th)
        b = torch.tensor(np.asarray(beta, dtype=np.float64), device=self.dev)[:, None]
        self.weight = self.sin * torch.sigmoid(-b * (E - mu)) * (SCALE / self.K)  # [B, K]
        self.bonds()

    def spinor(self, s):
        h = 0.5 * s[..., 0]
        return torch.stack([torch.complex(torch.cos(h), torch.zeros_like(h)),
                            torch.polar(torch.sin(h), s[..., 1])], -1)

    def bonds(self):
        chi = self.spinor(self.spins)
        self.h = -(chi[:, None].conj() * chi[:, self.nb]).sum(-1) / SCALE  # [B, 6, N]

    def recursion(self, r0, sites):
        """<l_j|T_n|r0> for n < M at the given sites: r0 [B, V, N] -> [B, V, M, len(sites)]."""
        h = self.h[:, None]
        out = torch.empty(r0.shape[:2] + (self.M, len(sites)), dtype=r0.dtype, device=self.dev)
        prev, cur = r0, (h * r0[:, :, self.nb]).sum(2)
        out[:, :, 0], out[:, :, 1] = prev[:, :, sites], cur[:, :, sites]
        for n in range(2, self.M):
            prev, cur = cur, 2 * (h * cur[:, :, self.nb]).sum(2) - prev
            out[:, :, n] = cur[:, :, sites]
        return out

    def sites(self, o):
        return torch.cat([torch.tensor([o], device=self.dev), self.nb[:, o]])

    def moments(self, o):
        loc = self.sites(o)
        r0 = torch.zeros(self.B, 7, self.N, dtype=torch.complex128, device=self.dev)
        r0[:, torch.arange(7, device=self.dev), loc] = 1
        return self.recursion(r0, loc).permute(0, 3, 1, 2)  # [B, j, k, n]

    def delta_omega(self, o, new):
        """Delta Omega [B] of moving the spin of o to new [B, 2]."""
        loc = self.sites(o)
        chi, chn = self.spinor(self.spins), self.spinor(new)
        v = -(chi[:, loc[1:]].conj() * (chn - chi[:, o])[:, None]).sum(-1) / SCALE  # Delta~ |o>, [B, 6]
        r0 = torch.zeros(self.B, 2, self.N, dtype=torch.complex128, device=self.dev)
        r0[:, 0, o] = 1
        r0[:, 1, loc[1:]] = v
        e = self.recursion(r0, loc)
        oo, ov = e[:, 0, :, 0].real + 0j, e[:, 1, :, 0]
        vv = (v.conj()[:, None] * e[:, 1, :, 1:]).sum(-1).real + 0j
        G = [m @ self.green.T for m in (oo, ov, ov.conj(), vv)]
        d = (1 + G[1]) * (1 + G[2]) - G[0] * G[3]
        arg = torch.angle(d)
        inc = arg[:, :-1] - arg[:, 1:]
        inc = inc - 2 * math.pi * (inc > math.pi) + 2 * math.pi * (inc <= -math.pi)
        phase = torch.flip(torch.cumsum(torch.flip(torch.cat([inc, arg[:, -1:]], 1), [1]), 1), [1])
        return (self.weight * phase).sum(1)

    def updates(self, n, seed, chain_ids, beta):
        dom, dec = [], []
        for u in range(n):
            o = u % self.N
            new, coin = [], []
            for c in chain_ids:
                x = _philox(seed & 0xFFFFFFFF, (seed >> 32) ^ c, u)
                new.append([math.acos(1 - 2 * x[0] * 2.0 ** -32), 2 * math.pi * x[1] * 2.0 ** -32])
                coin.append(((x[2] >> 5) * 67108864.0 + (x[3] >> 6)) * 2.0 ** -53)
            new = torch.tensor(new, device=self.dev, dtype=torch.float64)
            d = self.delta_omega(o, new)
            acc = np.exp(-np.asarray(beta) * d.cpu().numpy()) > np.array(coin)
            dom.append(d.cpu().numpy())
            dec.append(acc)
            a = torch.tensor(acc, device=self.dev)[:, None]
            self.spins[:, o] = torch.where(a, new, self.spins[:, o])
            self.bonds()
        return np.stack(dom, 1), np.stack(dec, 1).astype(np.uint8)


def exact(case, seed):
    if case["call"] in ("batch", "plan"):
        Ls, betas, spins = _members(case, seed)
        order = sorted(range(len(Ls)), key=lambda c: -Ls[c]) if case["call"] == "plan" else list(range(len(Ls)))
        dom = {}
        for L in sorted(set(Ls)):
            ids = [c for c in range(len(Ls)) if Ls[c] == L]
            sim = _Exact(L, np.stack([spins[c] for c in ids]), case["M"], betas[ids], case["mu"])
            d, _ = sim.updates(case["updates"], 1 + seed, ids, betas[ids])
            dom.update(zip(ids, d))
        return {"d_omega": np.concatenate([dom[c] for c in order]), "decisions": None, "n_accepted": None}
    sim = _Exact(case["L"], _spins(case, case["L"], seed)[None], case["M"], [case["beta"]], case["mu"],
                 case["kernel"], case["nodes"])
    o, th, ph = _probe(case, seed)
    if case["call"] == "moments":
        return sim.moments(o)[0].cpu().numpy()
    if case["call"] == "delta_omega":
        return sim.delta_omega(o, torch.tensor([[th, ph]], device=sim.dev, dtype=torch.float64)).cpu().numpy()
    d, _ = sim.updates(case["updates"], 1 + seed, [0], [case["beta"]])
    return {"d_omega": d[0], "decisions": None, "spins": sim.spins[0].cpu().numpy()}
