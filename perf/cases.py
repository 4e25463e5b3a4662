"""What a user of this framework has it do, as cases that can be timed.

Every case goes through the public entry points (``SwapSystem``, ``SwapBatch``,
``autodiff`` and the C-ABI binding's device read-outs).  The kinds:

* ``md``: dynamics of one system, then its state, its energies and (``log``)
  the per-step energy records are read;
* ``batch``: dynamics of many systems in one launch, then every state is read;
* ``forces``: forces and energies at positions an outer program supplies
  (a minimiser, a Monte-Carlo move, another integrator);
* ``diff``: energies, forces and the force-matching gradient with respect to
  (lambda, eps, sigma) over a batch of snapshots.

Results of FP32 systems carry single precision and are returned as float32 (as
a trajectory file stores them); FP64 systems return float64.  ``exact`` is a
plain torch restatement in 64 bits: dense neighbour rows, velocity Verlet or
BAOAB with Philox4x32-10 noise.

Runs are short (10 to 100 steps a pass): molecular trajectories are chaotic,
and two runs can be compared value by value only while they are.
"""
import math

import numpy as np
import torch

from paper_1912_08569_gb300 import SwapBatch, SwapSystem, autodiff
from paper_1912_08569_gb300 import _abi as A

GAMMA, DT, SKIN = 1.0, 0.001, 0.3


# --------------------------------------------------------------------------
# The cases

def listed():
    return [
        # the paper's timing system (section "Performance") at its smallest size:
        # launches and the chain of dependent phases of a step are what counts
        dict(name="dumbbell512", kind="md", mix="dumbbell", precision="fp32", n=512, density=0.125, n_exp=100,
             rcut=1.3, lambda3=1.0, shift=0, kT=0.03, gamma=GAMMA, steps=64, log=0),
        # the same system in the middle of the paper's range of sizes
        dict(name="dumbbell16k", kind="md", mix="dumbbell", precision="fp32", n=16384, density=0.125, n_exp=100,
             rcut=1.3, lambda3=1.0, shift=0, kT=0.03, gamma=GAMMA, steps=64, log=0),
        # a small ragged system with three types, two reactive pairs of different
        # coefficients and the continuous (shifted) form: no uniform coefficients
        dict(name="ternary4099", kind="md", mix="ternary", precision="fp32", n=4099, density=0.4, n_exp=10,
             rcut=1.5, lambda3=2.0, shift=1, kT=0.1, gamma=GAMMA, steps=100, log=0),
        # the throughput workload: dense binary mixture, Langevin, every step logged
        dict(name="mix100k", kind="md", mix="binary", precision="fp32", n=100_000, density=0.5, n_exp=10,
             rcut=1.5, lambda3=1.0, shift=0, kT=0.05, gamma=GAMMA, steps=100, log=1),
        # a system far larger than on-chip memory
        dict(name="mix1m", kind="md", mix="binary", precision="fp32", n=1_000_000, density=0.5, n_exp=10,
             rcut=1.5, lambda3=1.0, shift=0, kT=0.05, gamma=GAMMA, steps=20, log=0),
        # the validation run: FP64, constant energy, every step logged
        dict(name="nve2k_fp64", kind="md", mix="binary", precision="fp64", n=2000, density=0.2, n_exp=10,
             rcut=1.5, lambda3=1.0, shift=0, kT=0.1, gamma=0.0, steps=100, log=1),
        # FP64 Langevin dynamics of a dense, strongly shielded mixture
        dict(name="mix20k_fp64", kind="md", mix="binary", precision="fp64", n=20_000, density=0.5, n_exp=10,
             rcut=1.5, lambda3=5.0, shift=0, kT=0.05, gamma=GAMMA, steps=40, log=0),
        # the bonded network: chains of 50 beads with swapping crosslinkers, two million beads
        dict(name="network2m", kind="md", mix="network", precision="fp32", n=1_999_965, density=0.85, n_exp=10,
             rcut=1.5, lambda3=1.0, shift=0, kT=0.5, gamma=GAMMA, steps=10, log=0),
        # a parameter sweep: independent systems of uneven size, coefficients and temperature
        dict(name="sweep96", kind="batch", precision="fp32", systems=96, n_min=1000, n_max=16000, steps=50),
        # one gradient of a force-matching fit
        dict(name="fit20k", kind="diff", precision="fp32", n=20_000, density=0.4, n_exp=10, rcut=1.5, snapshots=16),
        # forces for an outer program: a call on a small system, and on a large one
        dict(name="forces1200", kind="forces", precision="fp32", n=1200, density=0.4, n_exp=10, rcut=1.5,
             lambda3=1.0, shift=0),
        dict(name="forces100k", kind="forces", precision="fp32", n=100_000, density=0.5, n_exp=10, rcut=1.5,
             lambda3=1.0, shift=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: sizes over their logarithm, options as the listed cases use them."""
    kind = rng.choice(["dumbbell", "binary", "binary", "ternary", "network", "fp64", "batch", "diff", "forces"])
    lam = rng.choice([0.0, 0.5, 1.0, 2.0, 5.0])
    if kind == "dumbbell":
        n = _log_int(rng, 512, 131_072)
        return dict(kind="md", mix="dumbbell", precision="fp32", n=n, density=0.125, n_exp=100,
                    rcut=rng.choice([1.15, 1.3]), lambda3=1.0, shift=0, kT=0.03, gamma=GAMMA,
                    steps=max(32, min(64, 8_000_000 // n)), log=0)
    if kind == "binary":
        n = _log_int(rng, 1000, 1_000_000)
        return dict(kind="md", mix="binary", precision="fp32", n=n, density=round(rng.uniform(0.2, 0.5), 3), n_exp=10,
                    rcut=1.5, lambda3=lam, shift=rng.choice([0, 0, 1]), kT=round(rng.uniform(0.05, 0.2), 3),
                    gamma=rng.choice([0.0, GAMMA]), steps=max(20, min(100, 10_000_000 // n)), log=rng.choice([0, 1, 10]))
    if kind == "ternary":
        n = _log_int(rng, 1000, 200_000)
        return dict(kind="md", mix="ternary", precision="fp32", n=n, density=round(rng.uniform(0.2, 0.5), 3), n_exp=10,
                    rcut=1.5, lambda3=lam, shift=1, kT=round(rng.uniform(0.05, 0.2), 3), gamma=GAMMA,
                    steps=max(20, min(100, 10_000_000 // n)), log=rng.choice([0, 1]))
    if kind == "network":
        n = 55 * _log_int(rng, 100, 36_363)
        return dict(kind="md", mix="network", precision="fp32", n=n, density=0.85, n_exp=10, rcut=1.5, lambda3=lam,
                    shift=0, kT=0.5, gamma=GAMMA, steps=max(10, min(100, 10_000_000 // n)), log=0)
    if kind == "fp64":
        n = _log_int(rng, 1000, 40_000)
        return dict(kind="md", mix="binary", precision="fp64", n=n, density=round(rng.uniform(0.2, 0.5), 3), n_exp=10,
                    rcut=1.5, lambda3=lam, shift=rng.choice([0, 1]), kT=round(rng.uniform(0.05, 0.2), 3),
                    gamma=rng.choice([0.0, GAMMA]), steps=max(20, min(100, 800_000 // n)), log=rng.choice([0, 1]))
    if kind == "batch":
        hi = _log_int(rng, 2000, 16_000)
        return dict(kind="batch", precision="fp32", systems=_log_int(rng, 8, 96), n_min=rng.choice([500, 1000]),
                    n_max=hi, steps=50)
    if kind == "diff":
        n = _log_int(rng, 2000, 32_000)
        return dict(kind="diff", precision=rng.choice(["fp32", "fp32", "fp64"]), n=n,
                    density=round(rng.uniform(0.3, 0.5), 3), n_exp=10, rcut=1.5, snapshots=rng.randint(2, 12))
    return dict(kind="forces", precision=rng.choice(["fp32", "fp32", "fp64"]), n=_log_int(rng, 400, 200_000),
                density=round(rng.uniform(0.2, 0.5), 3), n_exp=10, rcut=1.5, lambda3=lam, shift=rng.choice([0, 1]))


# --------------------------------------------------------------------------
# Inputs, from the seed alone

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _generator(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) * 1_000_003 + 17)
    return g


def _f32(t):
    return t.to(torch.float32).to(torch.float64)


def _edge(n, density):
    return float(np.float32((n / density) ** (1.0 / 3.0)))


class _Accepted:
    """Random sequential addition of objects of p points: a grid of cells that
    hold one point at most, checked 125 cells around every candidate point."""

    def __init__(self, L, sep):
        dev = _device()
        self.L, self.sep = L, sep
        self.m = int(math.ceil(L * math.sqrt(3.0) / sep))
        assert self.m <= int(2.0 * L / sep) and self.m >= 5, "box too small for the separation"
        self.owner = torch.full((self.m ** 3,), -1, dtype=torch.int64, device=dev)
        self.pts = torch.empty((0, 3), dtype=torch.float64, device=dev)
        r = torch.arange(-2, 3, device=dev)
        self.around = torch.stack(torch.meshgrid(r, r, r, indexing="ij"), -1).reshape(1, -1, 3)

    def _near(self, P, own, pts, limit):
        """Whether a point of `pts` (found through the cells `own`, of an index below `limit`) is within sep of each of P."""
        c = torch.remainder(torch.clamp((P / self.L * self.m).long(), max=self.m - 1)[:, None, :] + self.around, self.m)
        q = own[(c[..., 2] * self.m + c[..., 1]) * self.m + c[..., 0]]
        if len(pts) == 0:
            return torch.zeros(len(P), dtype=torch.bool, device=P.device)
        d = pts[q.clamp(min=0)] - P[:, None, :]
        d -= self.L * torch.round(d / self.L)
        hit = (q >= 0) & ((d * d).sum(-1) < self.sep * self.sep)
        if limit is not None:
            hit &= q < limit[:, None]
        return hit.any(1)

    def add(self, cand, want):
        """The first `want` of the candidates [M, p, 3] that fit (each against the points so far and earlier candidates)."""
        M, p = cand.shape[:2]
        flat = cand.reshape(-1, 3)
        old = self._near(flat, self.owner, self.pts, None)
        keep = ~old.reshape(M, p).any(1)
        cand = cand[keep]
        M = len(cand)
        if M == 0:
            return cand
        flat = cand.reshape(-1, 3)
        idx = torch.arange(M * p, device=flat.device)
        c = torch.clamp((flat / self.L * self.m).long(), max=self.m - 1)
        cell = (c[:, 2] * self.m + c[:, 1]) * self.m + c[:, 0]
        own = torch.full_like(self.owner, M * p).scatter_reduce_(0, cell, idx, "amin", include_self=True)
        lost = own[cell] != idx  # an earlier candidate's point is in the same cell
        own[own == M * p] = -1
        bad = lost | self._near(flat, own, flat, (idx // p) * p)
        cand = cand[~bad.reshape(M, p).any(1)][:want]
        flat = cand.reshape(-1, 3)
        c = torch.clamp((flat / self.L * self.m).long(), max=self.m - 1)
        self.owner[(c[:, 2] * self.m + c[:, 1]) * self.m + c[:, 0]] = torch.arange(
            len(self.pts), len(self.pts) + len(flat), device=flat.device)
        self.pts = torch.cat([self.pts, flat])
        return cand

    def fill(self, count, make):
        left = count
        for _ in range(4000):
            if left == 0:
                return
            left -= len(self.add(make(min(200_000, max(256, 3 * left))), left))
        raise RuntimeError("random sequential addition did not finish")


def _uniform(m, L, g):
    x = _f32(torch.rand((m, 3), generator=g, device=_device(), dtype=torch.float64) * L)
    x[(x >= L) | (x < 2.0 ** -20)] = 0.0
    return x


def _maxwell(n, kT, g):
    v = torch.randn((n, 3), generator=g, device=_device(), dtype=torch.float64) * math.sqrt(kT)
    return _f32(v - v.mean(0))


def _swap(case, lam):
    n = case["n_exp"]
    rbond = ((1.0 - math.sqrt(0.5)) / 2.0) ** (-1.0 / n)
    return dict(kind=2, eps=1.0, sigma=1.0, n=n, rcut=case["rcut"], lambda3=lam, shift=case.get("shift", 0), rbond=rbond)


def _wca():
    return dict(kind=1, eps=1.0, sigma=1.0, n=6)


def _system_inputs(case, seed):
    """Box, positions, velocities, types, pair table and bonds of one system."""
    g = _generator(seed)
    n, mix = case["n"], case.get("mix", "binary")
    L = _edge(n, case["density"])
    dev = _device()
    w = dict(n=n, L=L, bonds=None, n_types=2, seed=int(seed) & 0x7FFFFFFF)
    if mix == "network":
        # chains of 50 beads followed by 5 free crosslinkers along a boustrophedon
        # path through a simple cubic lattice, 5 beads of each chain reactive
        m = int(math.ceil(n ** (1.0 / 3.0) - 1e-9))
        k = torch.arange(n, device=dev)
        z, y, x = k // (m * m), (k // m) % m, k % m
        y = torch.where(z % 2 == 0, y, m - 1 - y)
        row = k // m
        x = torch.where(row % 2 == 0, x, m - 1 - x)
        w["x"] = _f32((torch.stack([x, y, z], -1).double() + 0.5) * (L / m))
        chains = n // 55
        types = torch.full((chains, 55), 2, dtype=torch.int32, device=dev)
        pick = torch.rand((chains, 50), generator=g, device=dev).argsort(1)[:, :5]
        types.scatter_(1, pick, 0)
        types[:, 50:] = 1
        w["types"] = types.reshape(-1)
        base = np.arange(chains, dtype=np.int32)[:, None] * 55 + np.arange(49, dtype=np.int32)[None, :]
        w["bonds"] = np.stack([base.reshape(-1), base.reshape(-1) + 1], 1)
        w["n_types"] = 3
        w["pairs"] = {(0, 1): _swap(case, case["lambda3"])}
        for a in range(3):
            for b in range(a, 3):
                w["pairs"].setdefault((a, b), _wca())
    elif mix == "dumbbell":
        # 3:2 A:B, every B bonded to its own A at the minimum of the pair potential
        nb = (2 * n) // 5
        acc = _Accepted(L, 1.0)
        rmin = 2.0 ** (1.0 / case["n_exp"])

        def pairs(m):
            a = _uniform(m, L, g)
            u = torch.randn((m, 3), generator=g, device=dev, dtype=torch.float64)
            b = _f32(torch.remainder(a + rmin * u / u.norm(dim=1, keepdim=True), L))
            b[b >= L] = 0.0
            return torch.stack([a, b], 1)

        acc.fill(nb, pairs)
        acc.fill(n - 2 * nb, lambda m: _uniform(m, L, g)[:, None, :])
        w["x"] = acc.pts
        types = torch.zeros(n, dtype=torch.int32, device=dev)
        types[1:2 * nb:2] = 1
        w["types"] = types
        w["pairs"] = {(0, 1): _swap(case, case["lambda3"]), (0, 0): _wca(), (1, 1): _wca()}
    else:
        acc = _Accepted(L, 0.9)
        acc.fill(n, lambda m: _uniform(m, L, g)[:, None, :])
        w["x"] = acc.pts
        k = 3 if mix == "ternary" else 2
        w["n_types"] = k
        w["types"] = (torch.arange(n, device=dev) % k).to(torch.int32)
        lam = case.get("lambda3", 1.0)
        w["pairs"] = {(0, 1): _swap(case, lam), (0, 0): _wca(), (1, 1): _wca()}
        if k == 3:
            w["pairs"][(0, 2)] = dict(_swap(case, 0.5 * lam), eps=0.7)
            w["pairs"][(1, 2)] = _wca()
            w["pairs"][(2, 2)] = _wca()
    w["v"] = _maxwell(n, case.get("kT", 0.05), g)
    return w


def _make_system(w, precision):
    s = SwapSystem(w["n"], w["n_types"], [w["L"]] * 3, w["pairs"], precision=precision, seed=w["seed"], skin=SKIN)
    if w["bonds"] is not None:
        s.set_bonds(w["bonds"], 100.0, 1.0)
    return s


def _sweep(case, seed):
    """Systems of a sweep: sizes log-uniform, densities, temperatures and lambda spread (sizes from the case alone)."""
    r = np.random.Generator(np.random.Philox(case["systems"]))
    out = []
    for k in range(case["systems"]):
        n = int(round(math.exp(r.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        rho, kT = round(float(r.uniform(0.2, 0.5)), 3), round(float(r.uniform(0.03, 0.2)), 3)
        sub = dict(n=n, density=rho, kT=kT, lambda3=(0.0, 0.5, 1.0, 2.0, 5.0)[k % 5], n_exp=10, rcut=1.5, shift=0)
        out.append((sub, int(seed) * 1000 + k))
    return out


def _out_dtype(case):
    return torch.float32 if case["precision"] == "fp32" else torch.float64


def prepare(case, seed):
    kind = case["kind"]
    dev = _device()
    st = dict(case=case, kind=kind, dtype=_out_dtype(case))
    if kind == "batch":
        subs = _sweep(case, seed)
        ws = [_system_inputs(c, sd) for c, sd in subs]
        st["systems"] = [_make_system(w, case["precision"]) for w in ws]
        for s, w in zip(st["systems"], ws):
            s.set_state(w["x"], w["v"], w["types"])
        st["kT"] = [c["kT"] for c, _ in subs]
        st["batch"] = SwapBatch(st["systems"])
        st["cuts"] = np.concatenate([[0], np.cumsum([w["n"] for w in ws])]).tolist()
        n = st["cuts"][-1]
        st["x"] = torch.empty((n, 3), dtype=torch.float64, device=dev)
        st["v"] = torch.empty((n, 3), dtype=torch.float64, device=dev)
        return st
    if kind == "diff":
        ws = [_system_inputs(case, int(seed) * 100 + k) for k in range(case["snapshots"])]
        s = _make_system(ws[0], case["precision"])
        for w in ws:  # the list is sized for the densest snapshot before the fit, which does not read back
            s.set_state(w["x"], None, w["types"])
            s.compute_forces()
        st["model"] = autodiff.SwapModel(s, ws[0]["pairs"], ws[0]["types"].cpu().numpy())
        st["X"] = torch.stack([w["x"] for w in ws])
        st["target"] = torch.stack([_Plain([w]).forces(w["x"], torch.tensor([1.0, 1.0, 1.0], device=dev, dtype=torch.float64))["F"]
                                    for w in ws])
        st["theta"] = torch.tensor(_THETA, dtype=torch.float64, device=dev)
        return st
    w = _system_inputs(case, seed)
    s = _make_system(w, case["precision"])
    st.update(s=s, w=w)
    st["x"] = torch.empty((w["n"], 3), dtype=torch.float64, device=dev)
    if kind == "md":
        s.set_state(w["x"], w["v"], w["types"])
        st["v"] = torch.empty((w["n"], 3), dtype=torch.float64, device=dev)
        st["img"] = torch.empty((w["n"], 3), dtype=torch.int32, device=dev)
        if case["log"]:
            s.set_thermo_log(case["log"], case["steps"] // case["log"])  # one pass of records
    return st


_THETA = (1.3, 0.9, 1.02)


# --------------------------------------------------------------------------
# One pass

def _energies(th, dtype):
    return torch.tensor([th["U2"], th["U3"], th["K"], *th["W"]], dtype=dtype)


def run(state):
    kind, case, dtype = state["kind"], state["case"], state["dtype"]
    if kind == "md":
        s = state["s"]
        s.run(case["steps"], DT, case["kT"], case["gamma"])
        A.swp_read_state(s.ctx, state["x"], state["v"], state["img"], where=A.SWP_DEVICE)
        th = s.thermo()
        out = dict(x=state["x"].to(dtype), v=state["v"].to(dtype), img=state["img"], energies=_energies(th, dtype),
                   bonds=th["n_bonds"], step=th["step"])
        if case["log"]:
            r = s.thermo_log()
            out["log"] = torch.from_numpy(np.column_stack([r["U2"], r["U3"], r["K"], r["W"]])).to(dtype)
            out["log_steps"] = r["step"]
            out["log_bonds"] = r["n_bonds"]
        return out
    if kind == "batch":
        state["batch"].run(case["steps"], DT, state["kT"], GAMMA)
        cuts = state["cuts"]
        for k, s in enumerate(state["systems"]):
            A.swp_read_state(s.ctx, state["x"][cuts[k]:cuts[k + 1]], state["v"][cuts[k]:cuts[k + 1]], None,
                             where=A.SWP_DEVICE)
        return dict(x=state["x"].to(dtype), v=state["v"].to(dtype))
    if kind == "diff":
        theta = state["theta"].clone().requires_grad_(True)
        X = state["X"].detach().requires_grad_(True)
        U = autodiff.energy_batch(state["model"], X, theta)
        (gX,) = torch.autograd.grad(U.sum(), X, create_graph=True)
        loss = ((gX + state["target"]) ** 2).mean()
        loss.backward()
        return dict(U=U.detach().to(dtype), gX=gX.detach().to(dtype), loss=loss.detach().to(dtype),
                    gtheta=theta.grad.to(dtype))
    s, w = state["s"], state["w"]
    s.set_state(w["x"], types=w["types"])
    s.compute_forces()
    A.swp_read_forces(s.ctx, state["x"], where=A.SWP_DEVICE)
    th = s.thermo()
    return dict(F=state["x"].to(dtype), energies=_energies(th, dtype), bonds=th["n_bonds"])


# --------------------------------------------------------------------------
# What a pass cannot do without

def _neighbours(case, density=None):
    """(reactive, other) partners of a particle inside the list radius."""
    rho = case.get("density", density)
    mix = case.get("mix", "binary")
    ball = lambda r: 4.0 / 3.0 * math.pi * r ** 3  # noqa: E731
    rs, rw = case.get("rcut", 1.5) + SKIN, 2.0 ** (1.0 / 6.0) + SKIN
    frac = {"binary": 0.5, "ternary": 4.0 / 9.0, "dumbbell": 0.48, "network": 0.0165}[mix]
    return rho * frac * ball(rs), rho * (1.0 - frac) * ball(rw)


def work(case):
    kind = case["kind"]
    # one pair: distance 11, potential and force 15, sums 6; the three-body factor 8;
    # a reactive pair's normalised potential once more for S: 28.  Integrator with noise: 150
    pair = lambda nr, nw: nr * (28 + 40) + nw * 32  # noqa: E731
    if kind == "batch":
        subs = [c for c, _ in _sweep(case, 0)]
        n = sum(c["n"] for c in subs)
        nr, nw = _neighbours(dict(density=0.35))
        return dict(bytes=float(n * case["steps"] * 80), flops=float(n * case["steps"] * (pair(nr, nw) + 150)))
    nr, nw = _neighbours(case)
    n = case["n"]
    if kind == "md":
        # position and velocity read and written once a step
        return dict(bytes=float(n * case["steps"] * 80), flops=float(n * case["steps"] * (pair(nr, nw) + 150)))
    # new positions: every pair inside the list radius has to be found (11 a candidate, about 6 candidates a pair)
    find = (nr + nw) * 6 * 11
    if kind == "forces":
        return dict(bytes=float(n * (24 + 4 + 24)), flops=float(n * (pair(nr, nw) + find)))
    m = n * case["snapshots"]
    # positions and targets in; forces, their derivatives (three parameters) and the gradient out
    return dict(bytes=float(m * (24 + 24 + 24 + 72 + 24)), flops=float(m * (pair(nr, nw) + find + nr * 2 * 60)))


# --------------------------------------------------------------------------
# The same in 64 bits, in plain torch

class _Plain:
    """Forces, energies and dynamics of independent systems (concatenated) over
    dense neighbour rows; `order` of sums fixed, so the values repeat."""

    def __init__(self, ws, gamma=0.0, kT=None):
        dev = _device()
        self.ws = ws
        self.cuts = np.concatenate([[0], np.cumsum([w["n"] for w in ws])]).tolist()
        self.n = self.cuts[-1]
        per = lambda vals: torch.cat([torch.full((w["n"], 1), float(v), dtype=torch.float64, device=dev)  # noqa: E731
                                      for w, v in zip(ws, vals)])
        self.L = per([w["L"] for w in ws])
        self.kT = None if kT is None else per(kT)
        self.seed = torch.cat([torch.full((w["n"],), w["seed"], dtype=torch.int64, device=dev) for w in ws])
        self.tag = torch.cat([torch.arange(w["n"], device=dev) for w in ws])
        self.gamma = gamma
        self.bond = None
        if ws[0]["bonds"] is not None:
            b = torch.from_numpy(ws[0]["bonds"]).to(dev).long()
            both = torch.cat([b, b.flip(1)])
            both = both[both[:, 0].argsort(stable=True)]
            cnt = torch.bincount(both[:, 0], minlength=self.n)
            at = torch.arange(len(both), device=dev) - (cnt.cumsum(0) - cnt)[both[:, 0]]
            self.bond = torch.full((self.n, 2), -1, dtype=torch.int64, device=dev)
            self.bond[both[:, 0], at] = both[:, 1]

    # neighbour rows -------------------------------------------------------
    def _rows_of(self, w, x, margin):
        """Dense rows of one system's partners inside the largest cut-off + margin."""
        dev, n, L = x.device, w["n"], w["L"]
        cut = max(p["rcut"] if p["kind"] == 2 else p["sigma"] * 2.0 ** (1.0 / p["n"]) for p in w["pairs"].values())
        rl = cut + margin
        m = max(3, int(L / rl))
        c = torch.clamp((torch.remainder(x, L) / L * m).long(), max=m - 1)
        cell = (c[:, 2] * m + c[:, 1]) * m + c[:, 0]
        order = cell.argsort(stable=True)
        cnt = torch.bincount(cell, minlength=m ** 3)
        start = cnt.cumsum(0) - cnt
        cap = int(cnt.max())
        table = torch.full((m ** 3, cap), -1, dtype=torch.int64, device=dev)
        sc = cell[order]
        table[sc, torch.arange(n, device=dev) - start[sc]] = order
        r = torch.arange(-1, 2, device=dev)
        around = torch.stack(torch.meshgrid(r, r, r, indexing="ij"), -1).reshape(1, -1, 3)
        rows, K = [], 0
        step = max(1, 40_000_000 // (27 * cap))
        for a in range(0, n, step):
            b = min(a + step, n)
            cc = torch.remainder(c[a:b, None, :] + around, m)
            cand = table[(cc[..., 2] * m + cc[..., 1]) * m + cc[..., 0]].reshape(b - a, -1)
            d = x[cand.clamp(min=0)] - x[a:b, None, :]
            d -= L * torch.round(d / L)
            ok = (cand >= 0) & ((d * d).sum(-1) < rl * rl) & (cand != torch.arange(a, b, device=dev)[:, None])
            del d
            k = int(ok.sum(1).max()) if b > a else 0
            out = torch.full((b - a, k), -1, dtype=torch.int64, device=dev)
            i, j = ok.nonzero(as_tuple=True)
            out[i, ok.cumsum(1)[i, j] - 1] = cand[i, j]
            rows.append(out)
            K = max(K, k)
        return torch.cat([torch.nn.functional.pad(o, (0, K - o.shape[1]), value=-1) for o in rows])

    def build(self, x, margin=0.4):
        dev = x.device
        rows = [self._rows_of(w, x[a:b], margin) for w, a, b in zip(self.ws, self.cuts, self.cuts[1:])]
        K = max(r.shape[1] for r in rows)
        J = torch.cat([torch.nn.functional.pad(torch.where(r >= 0, r + a, r), (0, K - r.shape[1]), value=-1)
                       for r, a in zip(rows, self.cuts)])
        self.ok = J >= 0
        self.J = J.clamp(min=0)
        # coefficients of every entry, by its pair of types
        names = ("swap", "eps", "sig2", "n", "rc2", "rmin2", "a2", "vshift", "ushift", "epshat")
        out = {k: [] for k in names}
        for w, a, b in zip(self.ws, self.cuts, self.cuts[1:]):
            t = w["n_types"]
            tab = torch.zeros((len(names), t * t), dtype=torch.float64)
            for (i, j), p in w["pairs"].items():
                sw = p["kind"] == 2
                rmin = p["sigma"] * 2.0 ** (1.0 / p["n"])
                rc = p["rcut"] if sw else rmin
                xc = (p["sigma"] / rc) ** p["n"]
                vc = 4.0 * p["eps"] * (xc * xc - xc) if sw and p["shift"] else 0.0
                vals = (float(sw), p["eps"], p["sigma"] ** 2, p["n"], rc * rc, rmin * rmin,
                        p["lambda3"] * p["eps"] if sw else 0.0, vc, -vc if sw else p["eps"], p["eps"] + vc)
                for q in (i * t + j, j * t + i):
                    tab[:, q] = torch.tensor(vals, dtype=torch.float64)
            ty = w["types"].long()
            at = ty[:, None] * t + ty[(self.J[a:b] - a).clamp(min=0)]
            tab = tab.to(dev)
            for k, name in enumerate(names):
                out[name].append(tab[k][at])
        self.c = {k: torch.cat(v) for k, v in out.items()}
        self.c["swap"] = self.c["swap"] > 0.5
        return self

    # forces ---------------------------------------------------------------
    def forces(self, x, theta=None, build=True):
        if build:
            self.build(x)
        c, J = self.c, self.J
        sw = c["swap"]
        eps, sig2, rmin2, a2, epshat, ush = c["eps"], c["sig2"], c["rmin2"], c["a2"], c["epshat"], c["ushift"]
        if theta is not None:  # (lambda, eps, sigma) of the reactive pair
            eps = torch.where(sw, theta[1], eps)
            sig2 = torch.where(sw, theta[2] ** 2, sig2)
            rmin2 = torch.where(sw, theta[2].detach() ** 2 * 2.0 ** (2.0 / c["n"]), rmin2)
            a2 = torch.where(sw, theta[0] * theta[1], a2)
            epshat = eps
        d = x[J] - x[:, None, :]
        d = d - self.L[:, :, None] * torch.round(d / self.L[:, :, None])
        r2 = torch.where(self.ok, (d * d).sum(-1), torch.full_like(c["n"], 1e6))
        inside = r2 < c["rc2"]
        q = (sig2 / r2) ** (0.5 * c["n"])
        v = 4.0 * eps * (q * q - q)
        f = 4.0 * eps * c["n"] * (2.0 * q * q - q) / r2
        beyond = r2 > rmin2
        a = torch.sqrt(a2)
        avh = torch.where(inside & sw, a * torch.where(beyond, (c["vshift"] - v) / epshat, torch.ones_like(v)),
                          torch.zeros_like(v))
        S = avh.sum(1)
        h = a * (S[:, None] + S[J] - 2.0 * avh)
        f = torch.where(inside, torch.where(sw & beyond, f * (1.0 - h / epshat), f), torch.zeros_like(f))
        F = -(f[..., None] * d).sum(1)
        u2 = torch.where(inside, 0.5 * (v + ush), torch.zeros_like(v)).sum(1)
        u3 = (0.5 * avh * (S[:, None] - avh)).sum(1)
        pick = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
        W = [0.5 * (f * d[..., i] * d[..., k]).sum() for i, k in pick]
        if self.bond is not None:
            for b in range(2):
                j = self.bond[:, b].clamp(min=0)
                has = self.bond[:, b] >= 0
                e = x[j] - x
                e = e - self.L * torch.round(e / self.L)
                r = e.norm(dim=1)
                g = torch.where(has, 100.0 * (r - 1.0) / r.clamp(min=1e-9), torch.zeros_like(r))
                F = F + g[:, None] * e
                u2 = u2 + torch.where(has, 25.0 * (r - 1.0) ** 2, torch.zeros_like(r))
                W = [t - 0.5 * (g * e[:, i] * e[:, k]).sum() for t, (i, k) in zip(W, pick)]
        return dict(F=F, u2=u2, u3=u3, W=torch.stack(W))

    # dynamics -------------------------------------------------------------
    def _normals(self, step):
        """Three normals a particle: Philox4x32-10 (Salmon et al., SC'11), counter (tag, step lo, step hi, 1), key = seed; Box-Muller."""
        M = 0xFFFFFFFF
        c = [self.tag, torch.full_like(self.tag, step & M), torch.full_like(self.tag, step >> 32), torch.ones_like(self.tag)]
        k0, k1 = self.seed & M, self.seed >> 32

        def mul(a, b):
            # 32 x 32 -> (high, low) through 16-bit halves of b: no product exceeds 63 bits
            lo, hi = a * (b & 0xFFFF), a * (b >> 16)
            t = (lo >> 16) + hi
            return (t >> 16) & M, ((t << 16) | (lo & 0xFFFF)) & M

        for _ in range(10):
            h0, l0 = mul(torch.full_like(self.tag, 0xD2511F53), c[0])
            h1, l1 = mul(torch.full_like(self.tag, 0xCD9E8D57), c[2])
            c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
            k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
        u = [(t.double() + 0.5) / 2.0 ** 32 for t in c]
        ra, rb = torch.sqrt(-2.0 * torch.log(u[0])), torch.sqrt(-2.0 * torch.log(u[2]))
        return torch.stack([ra * torch.cos(2 * math.pi * u[1]), ra * torch.sin(2 * math.pi * u[1]),
                            rb * torch.cos(2 * math.pi * u[3])], 1)

    def dynamics(self, x, v, steps, record=()):
        """x (wrapped), v, forces after `steps` steps of unit-mass particles, and the energies of the steps in `record`."""
        h = 0.5 * DT
        r = self.forces(x)
        log = {}
        c1 = math.exp(-self.gamma * DT)
        for k in range(steps):
            v = v + h * r["F"]
            x = x + h * v
            if self.gamma > 0.0:
                v = c1 * v + torch.sqrt((1.0 - c1 * c1) * self.kT) * self._normals(k)
            x = torch.remainder(x + h * v, self.L)
            r = self.forces(x, build=(k + 1) % 10 == 0)
            v = v + h * r["F"]
            if k + 1 in record:
                log[k + 1] = self.energies(r, v)
        return x, v, r, log

    @staticmethod
    def energies(r, v):
        e = torch.stack([r["u2"].sum(), r["u3"].sum(), 0.5 * (v * v).sum()])
        return torch.cat([e, r["W"]])


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        subs = _sweep(case, seed)
        ws = [_system_inputs(c, sd) for c, sd in subs]
        p = _Plain(ws, GAMMA, [c["kT"] for c, _ in subs])
        x, v, _, _ = p.dynamics(torch.cat([w["x"] for w in ws]), torch.cat([w["v"] for w in ws]), case["steps"])
        return dict(x=x, v=v)
    if kind == "diff":
        dev = _device()
        theta = torch.tensor(_THETA, dtype=torch.float64, device=dev, requires_grad=True)
        U, gX, loss = [], [], 0.0
        for k in range(case["snapshots"]):
            w = _system_inputs(case, int(seed) * 100 + k)
            p = _Plain([w])
            target = p.forces(w["x"], torch.tensor([1.0, 1.0, 1.0], device=dev, dtype=torch.float64))["F"]
            r = p.forces(w["x"], theta, build=False)
            part = ((target - r["F"]) ** 2).mean() / case["snapshots"]
            part.backward()
            loss = loss + part.detach()
            U.append((r["u2"].sum() + r["u3"].sum()).detach())
            gX.append(-r["F"].detach())
        return dict(U=torch.stack(U), gX=torch.stack(gX), loss=loss, gtheta=theta.grad)
    w = _system_inputs(case, seed)
    if kind == "forces":
        r = _Plain([w]).forces(w["x"])
        e = _Plain.energies(r, torch.zeros_like(w["v"]))
        return dict(F=r["F"], energies=e, bonds=None)
    p = _Plain([w], case["gamma"], [case["kT"]])
    record = set(range(case["log"], case["steps"] + 1, case["log"])) if case["log"] else set()
    x, v, r, log = p.dynamics(w["x"], w["v"], case["steps"], record)
    out = dict(x=x, v=v, img=None, energies=p.energies(r, v), bonds=None, step=None)
    if case["log"]:
        out["log"] = torch.stack([log[k] for k in sorted(log)])
        out["log_steps"] = None
        out["log_bonds"] = None
    return out
