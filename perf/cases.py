"""Measured workloads of the SDPD library and their float64 reference values.

A case is one call pattern of a user's program on one system: full time steps
(Velocity Verlet and the fluctuation/dissipation sweep), Verlet steps alone,
sweeps alone with their energy histogram, a step with host buffers in and out,
an ensemble of replicas in one CUDA graph, a gradient.  ``listed()`` names the
fixed ones, ``draw(rng)`` gives one more of the same ranges, ``prepare`` makes
a case's handle and inputs from a seed, ``run`` is one pass through the public
entry points, ``work`` the bytes and operations a pass cannot do without, and
``exact`` the same pass in plain torch float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1707_04232_gb300 import sdpd
from paper_1707_04232_gb300.autograd import handle_theta, verlet_trajectory, virial_pressure
from paper_1707_04232_gb300.inputs import Workload, lattice_state, random_box_state

SCHEMES = {"ssa": sdpd.SCHEME_SSA, "ams": sdpd.SCHEME_AMS, "ems": sdpd.SCHEME_EMS, "none": sdpd.SCHEME_NONE}
KERNELS = {"lucy": sdpd.KERNEL_LUCY, "cubic": sdpd.KERNEL_CUBIC}
PRECISIONS = {"fp64": sdpd.FP64, "mixed": sdpd.MIXED}

# Every case has these keys.  kind: steps (state after `steps` full steps, and
# the observables), fd (sweeps at fixed positions and the energy histogram),
# host (one state loaded from pinned host memory, stepped and read back),
# ensemble (replicas of growing size in one graph), gradient (virial pressure
# after `steps` steps, differentiated).  layout: lattice (n^3 sites) or random
# (unit density in an lx x ly x lz box).
_BASE = {"kind": "steps", "layout": "lattice", "n": 10, "lx": 0.0, "ly": 0.0, "lz": 0.0, "precision": "fp64",
         "scheme": "ems", "kernel": "lucy", "K": 100.0, "kT": 1.0, "theta": 1, "dt": 0.005, "steps": 1,
         "replicas": 1, "n_max": 0, "sweep_f32": False}


def _case(**kw):
    return {**_BASE, **kw}


def listed():
    return [
        # the smallest call: Velocity Verlet alone on the paper's 1000
        # particles, its "Verlet" timing row; launches and gaps count
        _case(name="verlet_1k_fp64", scheme="none", steps=20),
        # the paper's own system size, full steps with the exact Metropolis
        # scheme, in the library's default precision
        _case(name="ems_1k_fp64", steps=4),
        # multiple time steps: ten small replicas in one graph, one sweep
        # every five Verlet steps (the energy-drift experiment)
        _case(name="mts_replicas_1k_fp64", kind="ensemble", K=5.0, theta=5, steps=10, replicas=10, n_max=10),
        # a disordered fluid in a rectangular box with an odd particle count,
        # cubic spline, approximate Metropolis scheme
        _case(name="ragged_3k_ams_cubic_fp64", layout="random", lx=12.5, ly=15.0, lz=17.3, kernel="cubic",
              scheme="ams", K=20.0, steps=3),
        # a side between two cell counts (14 / 2.5 = 5.6 cells, of which an
        # even number fits): cells of 3.5, so the 2x2x2 blocks hold 343
        _case(name="odd_side_2744_mixed", n=14, precision="mixed", steps=2),
        # ordinary size, mixed precision
        _case(name="ems_32k_mixed", n=32, precision="mixed", steps=4),
        # the same system in float64
        _case(name="ems_32k_fp64", n=32, steps=2),
        # sweeps alone at K = 5 with the energy histogram after them (the
        # distribution experiment): the schedule is built once and reused
        _case(name="fd_262k_mixed", kind="fd", n=64, precision="mixed", K=5.0, dt=0.22, steps=4),
        # cold K = 5 stress fluid stepped by a host program that owns the state
        _case(name="host_262k_mixed", kind="host", n=64, precision="mixed", K=5.0, kT=0.1),
        # the headline: one large fluid, mixed precision
        _case(name="ems_2m_mixed", n=128, precision="mixed", K=50.0, steps=2),
        # replicas of uneven size (13^3 .. 40^3, moved off the sizes whose
        # blocks overflow) in one graph
        _case(name="ensemble_mixed", kind="ensemble", precision="mixed", K=20.0, steps=4, replicas=24, n_max=40),
        # gradient of the virial pressure through recorded full steps
        _case(name="gradient_32k", kind="gradient", n=32, sweep_f32=True, steps=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "fd", "host", "ensemble", "gradient"])
    kernel = rng.choice(["lucy", "cubic"])
    if kind == "steps":
        precision = rng.choice(["fp64", "mixed"])
        scheme = rng.choice(["ems", "ems", "ams", "ssa", "none"])
        K = rng.choice([50.0, 100.0]) if scheme == "ssa" else rng.choice([5.0, 20.0, 50.0, 100.0])
        top = 100 if precision == "mixed" else 40
        c = dict(kind=kind, precision=precision, scheme=scheme, K=K, kernel=kernel, theta=rng.choice([1, 1, 2]))
        if rng.random() < 0.6:
            c["n"] = _log_int(rng, 10, top)
        else:
            s = math.exp(rng.uniform(math.log(11.0), math.log(0.8 * top)))
            c.update(layout="random", lx=round(s, 2), ly=round(s * rng.uniform(1.0, 1.25), 2),
                     lz=round(s * rng.uniform(1.0, 1.25), 2))
        c["steps"] = 2 * rng.choice([1, 2]) if precision == "mixed" or c.get("n", 99) < 16 else 2
        return _case(**c)
    if kind == "fd":
        K = rng.choice([5.0, 20.0, 100.0])
        return _case(kind=kind, n=_log_int(rng, 16, 80), precision="mixed", K=K, kernel=kernel,
                     scheme=rng.choice(["ems", "ams"]), dt=rng.choice([0.05, 0.22, 0.45]), steps=rng.choice([2, 3, 4]))
    if kind == "host":
        return _case(kind=kind, n=_log_int(rng, 16, 96), precision="mixed", kernel=kernel, K=rng.choice([5.0, 50.0]),
                     kT=rng.choice([0.1, 1.0]))
    if kind == "ensemble":
        if rng.random() < 0.4:
            return _case(kind=kind, K=5.0, theta=5, steps=10, replicas=rng.randint(4, 16), n_max=10, kernel=kernel)
        return _case(kind=kind, precision="mixed", K=rng.choice([5.0, 20.0, 100.0]), steps=rng.choice([2, 4]),
                     replicas=rng.randint(8, 24), n_max=rng.randint(16, 40), kernel=kernel)
    return _case(kind=kind, n=rng.randint(15, 32), sweep_f32=rng.random() < 0.7, kernel=kernel,
                 K=rng.choice([20.0, 100.0]), steps=rng.randint(3, 8))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _box(case):
    if case["layout"] == "lattice":
        return (float(case["n"]),) * 3
    return (case["lx"], case["ly"], case["lz"])


def _count(case):
    b = _box(case)
    return case["n"] ** 3 if case["layout"] == "lattice" else int(round(b[0] * b[1] * b[2]))


def _state(case, seed):
    """(q, p, eps) of the case's system, float64 in id order, host arrays."""
    if case["layout"] == "lattice":
        return lattice_state(Workload(n=case["n"], K=case["K"], kT=case["kT"], seed=seed))
    L = np.array(_box(case))
    q, p, e = random_box_state(_count(case), 1.0, 1.0, case["kT"], 1.5 * (case["K"] - 1.0) * case["kT"], seed=seed)
    q = q * L
    return np.where(q >= L, 0.0, q), p, e


def _handle(case, N, box, **kw):
    return sdpd.SDPD(N, box, m=1.0, h=2.5, K=case["K"], precision=PRECISIONS[case["precision"]],
                     scheme=SCHEMES[case["scheme"]], kernel=KERNELS[case["kernel"]], theta=case["theta"], **kw)


def _replica_sides(case):
    """Lattice sides of an ensemble's replicas: equal, or spread evenly over
    the logarithm of [13, n_max], each moved up to a side whose 2x2x2 cell
    blocks stay below 200 particles."""
    if case["n_max"] <= 13:
        return [case["n_max"]] * case["replicas"]
    out = []
    for k in range(case["replicas"]):
        n = int(round(13.0 * (case["n_max"] / 13.0) ** (k / max(1, case["replicas"] - 1))))
        while (2.0 * n / (int(n / 2.5) // 2 * 2)) ** 3 > 200.0:
            n += 1
        out.append(n)
    return out


def _out(N):
    return (torch.empty((N, 3), dtype=torch.float64, device="cuda"),
            torch.empty((N, 3), dtype=torch.float64, device="cuda"),
            torch.empty(N, dtype=torch.float64, device="cuda"))


def prepare(case, seed):
    st = {"case": case, "seed": seed & 0xFFFFFF}
    if case["kind"] == "ensemble":
        members, spans, at = [], [], 0
        for k, n in enumerate(_replica_sides(case)):
            w = Workload(n=n, K=case["K"], kT=case["kT"], seed=seed + 1000 * k)
            m = _handle(case, w.N, w.L, stream=torch.cuda.Stream())
            m.set_state(*lattice_state(w))
            members.append(m)
            spans.append((at, at + w.N))
            at += w.N
        st.update(ens=sdpd.SDPDEnsemble(members), members=members, spans=spans, out=_out(at),
                  seeds=[st["seed"] + k for k in range(len(members))])
        return st
    N = _count(case)
    q, p, e = _state(case, seed)
    if case["kind"] == "gradient":
        st["sim"] = _handle(case, N, _box(case), sweep_f32=case["sweep_f32"])
        st["x"] = [torch.as_tensor(a, device="cuda").requires_grad_() for a in (q, p, e)]
        st["theta"] = torch.tensor(handle_theta(st["sim"]), dtype=torch.float64, requires_grad=True)
        return st
    s = st["sim"] = _handle(case, N, _box(case), fd_only=case["kind"] == "fd")
    if case["kind"] == "host":
        st["host_in"] = [torch.from_numpy(a).pin_memory().numpy() for a in (q, p, e)]
        st["host_out"] = [torch.empty(a.shape, dtype=torch.float64, pin_memory=True).numpy() for a in (q, p, e)]
        return st
    s.set_state(q, p, e)
    st["out"] = _out(N)
    if case["kind"] == "fd":
        st["counts"] = torch.zeros(152, dtype=torch.int64, device="cuda")
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(st):
    case, kind = st["case"], st["case"]["kind"]
    dt, steps, seed = case["dt"], case["steps"], st["seed"]
    if kind == "ensemble":
        st["ens"].step(dt, steps, st["seeds"])
        q, p, e = st["out"]
        for m, (a, b) in zip(st["members"], st["spans"]):
            m.get_state_device(q[a:b], p[a:b], e[a:b])
        return {"q": q, "p": p, "eps": e}
    s = st["sim"]
    if kind == "gradient":
        q, p, e = st["x"]
        for t in (q, p, e, st["theta"]):
            t.grad = None
        x = verlet_trajectory(s, q, p, e, st["theta"], dt, steps, every=max(1, steps // 2), seed=seed)
        loss = virial_pressure(s, *x, st["theta"])
        loss.backward()
        return {"loss": loss.detach(), "gq": q.grad, "gp": p.grad, "geps": e.grad, "gtheta": st["theta"].grad}
    if kind == "host":
        q, p, e = st["host_in"]
        oq, op, oe = st["host_out"]
        s.set_state(q, p, e)
        s.step(dt, steps, seed=seed)
        status = sdpd.sdpd_get_state(s.h, oq.ctypes.data, op.ctypes.data, oe.ctypes.data, 0)
        return {"q": oq, "p": op, "eps": oe, "status": status}
    s.step(dt, steps, seed=seed)
    q, p, e = st["out"]
    if kind == "fd":
        st["counts"].zero_()
        s.energy_histogram(0.1, 20.0, 150, 1.0 / case["kT"], st["counts"])
        s.get_state_device(q, p, e)
        return {"p": p, "eps": e, "counts": st["counts"]}
    s.get_state_device(q, p, e)
    o = s.observables()
    return {"q": q, "p": p, "eps": e, "E": o["E"], "T_kin": o["T_kin"], "T_int": o["T_int"],
            "n_pairs": int(o["n_pairs"]), "n_reject": int(o["n_reject_bound"] + o["n_reject_metropolis"])}


def work(case):
    """State read and written once in its stored precision and the float64
    results written once (and the host inputs read); operations of the method:
    18 per density visit, 24 per force visit (two force passes), 210 / 150 /
    140 per EMS / AMS / SSA pair update, 23 + 66 per visit of the reverse
    passes."""
    kind = case["kind"]
    N = sum(n ** 3 for n in _replica_sides(case)) if kind == "ensemble" else _count(case)
    state = 112.0 if case["precision"] == "fp64" else 64.0
    nbr = 80.0 if case["layout"] == "lattice" else 65.4
    pair = {"ems": 210.0, "ams": 150.0, "ssa": 140.0, "none": 0.0}[case["scheme"]] * 0.5 * nbr
    verlet = 0.0 if kind == "fd" else nbr * (18.0 + 2 * 24.0)
    flops = N * case["steps"] * (verlet + pair / (1 if kind == "fd" else case["theta"]))
    nbytes = N * (state + 56.0 + (56.0 if kind in ("host", "gradient") else 0.0))
    if kind == "gradient":
        flops += N * (case["steps"] + 1) * nbr * 89.0
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# The same pass in plain torch float64
# ---------------------------------------------------------------------------

class _Ref:
    """Smoothed dissipative particle dynamics of an ideal gas, unit mass and
    kB = 1: density and forces from a pair list found by brute force, Velocity
    Verlet at fixed entropies, and the pairwise sweep in the library's
    documented order (8 cell-parity colours; in a 2x2x2 block of cells by
    rank difference, then lower rank) with Philox4x64-10 numbers."""

    def __init__(self, case, box, seed):
        self.case, self.seed, self.h = case, seed, 2.5
        self.L = torch.tensor(box, dtype=torch.float64, device="cuda")
        self.nc = torch.tensor([int(b / 2.5) // 2 * 2 for b in box], device="cuda")
        K = case["K"]
        self.CK, self.cr = 1.5 * (K - 1.0), 0.5 * (K - 1.0)
        self.lucy = case["kernel"] == "lucy"
        self.sweeps, self.n_pairs, self.n_reject = 0, 0, 0

    def W(self, r, h):
        x = r / h
        if self.lucy:
            return 105.0 / (16.0 * math.pi) / h ** 3 * (1 + 3 * x) * (1 - x) ** 3
        return 8.0 / math.pi / h ** 3 * torch.where(x <= 0.5, 1 - 6 * x * x + 6 * x ** 3, 2 * (1 - x) ** 3)

    def F(self, r, h):
        x = r / h
        if self.lucy:
            return 315.0 / (4.0 * math.pi) / h ** 5 * (1 - x) ** 2
        return 48.0 / math.pi / h ** 5 * torch.where(x <= 0.5, 2 - 3 * x, (1 - x) ** 2 / x.clamp_min(1e-9))

    def pairs(self, q):
        """Index pairs i < j with r_ij < h."""
        n = len(q)
        rows = max(1, min(n, (1 << 26) // n))
        out = []
        for a in range(0, n, rows):
            r2 = torch.zeros((min(rows, n - a), n - a), dtype=torch.float64, device="cuda")
            for k in range(3):
                d = (q[a:a + rows, None, k] - q[None, a:, k]).abs_()
                d = torch.minimum(d, self.L[k] - d)
                r2 += d * d
            i, j = torch.nonzero(r2 < self.h * self.h, as_tuple=True)
            keep = j > i
            out.append(torch.stack([i[keep], j[keep]]) + a)
        return torch.cat(out, 1)

    def disp(self, q, ij):
        d = q[ij[0]] - q[ij[1]]
        return d - self.L * torch.round(d / self.L).detach()

    def dist(self, d):
        return (d * d).sum(1).clamp_min(1e-300).sqrt()

    def density(self, q, ij, h):
        w = self.W(self.dist(self.disp(q, ij)), h)
        zero = torch.zeros(1, dtype=torch.float64, device="cuda")
        return self.W(zero, h) + torch.zeros(len(q), dtype=torch.float64, device="cuda").index_add(0, ij[0], w).index_add(0, ij[1], w)

    def force(self, q, rho, eps, ij, th):
        h, cr, CK = th
        pi = cr * eps / (CK * rho)
        d = self.disp(q, ij)
        f = ((pi[ij[0]] + pi[ij[1]]) * self.F(self.dist(d), h))[:, None] * d
        return torch.zeros_like(q).index_add(0, ij[0], f).index_add(0, ij[1], -f), d, f

    def verlet(self, q, p, eps, dt, th, ij=None):
        """One Velocity Verlet step; returns the new pair list too."""
        h, cr, CK = th
        ij = self.pairs(q.detach()) if ij is None else ij
        rho = self.density(q, ij, h)
        S = CK * torch.log(eps) - cr * torch.log(rho)
        p = p + 0.5 * dt * self.force(q, rho, eps, ij, th)[0]
        q = q + dt * p
        q = q - self.L * torch.floor(q / self.L).detach()
        ij = self.pairs(q.detach())
        rho = self.density(q, ij, h)
        eps = torch.exp((S + cr * torch.log(rho)) / CK)
        p = p + 0.5 * dt * self.force(q, rho, eps, ij, th)[0]
        return q, p, eps, ij

    # -- the sweep ----------------------------------------------------------

    @staticmethod
    def _mulhi(a, m):
        """High and low words of the unsigned product of a with the constant m."""
        mask, shr = 0xFFFFFFFF, lambda x, s: (x >> s) & ((1 << (64 - s)) - 1)
        al, ah, ml, mh = a & mask, shr(a, 32), m & mask, (m >> 32) & mask
        lo = al * ml
        mid = ah * ml + shr(lo, 32)
        mid2 = al * mh + (mid & mask)
        return ah * mh + shr(mid, 32) + shr(mid2, 32), (mid2 << 32) | (lo & mask)

    def randoms(self, i, j):
        """Three standard normals and one uniform per pair."""
        signed = lambda v: v - (1 << 64) if v >> 63 else v  # noqa: E731
        c = [torch.full_like(i, self.sweeps), i.clone(), j.clone(), torch.zeros_like(i)]
        k = [self.seed, 0]
        for _ in range(10):
            h0, l0 = self._mulhi(c[0], 0xD2E7470EE14C6C93)
            h1, l1 = self._mulhi(c[2], 0xCA5A826395121157)
            c = [h1 ^ c[1] ^ signed(k[0]), l1, h0 ^ c[3] ^ signed(k[1]), l0]
            k = [(k[0] + 0x9E3779B97F4A7C15) % 2 ** 64, (k[1] + 0xBB67AE8584CAA73B) % 2 ** 64]
        u53 = lambda w: (((w >> 11) & ((1 << 53) - 1)).double() + 0.5) * 2.0 ** -53  # noqa: E731
        u32 = lambda w: ((w & 0xFFFFFFFF).double() + 0.5) * 2.0 ** -32  # noqa: E731
        R, a = torch.sqrt(-2.0 * torch.log(u53(c[0]))), 2.0 * math.pi * u53(c[1])
        G2 = torch.sqrt(-2.0 * torch.log(u32(c[2] >> 32))) * torch.cos(2.0 * math.pi * u32(c[2]))
        return torch.stack([R * torch.cos(a), R * torch.sin(a), G2], 1), u53(c[3])

    def schedule(self, q, ij):
        """Per colour: the pairs' positions in ij, level by level."""
        nc = self.nc
        cell = torch.minimum(torch.floor(q / (self.L / nc)).long().clamp_min(0), nc - 1)
        i, j = ij
        x = i.clone()
        for mul, sh in ((2654435761, 15), (2246822519, 13), (3266489917, 16)):
            x = (x * mul) & 0xFFFFFFFF
            x = x ^ (x >> sh)
        bits = x >> 29
        own = []
        for k in range(3):
            a, b, b_k = cell[i, k], cell[j, k], (bits >> k) & 1
            own.append(torch.where(a == b, (a - b_k) % nc[k], torch.where((a + 1) % nc[k] == b, a, b)))
        colour = (own[0] & 1) | ((own[1] & 1) << 1) | ((own[2] & 1) << 2)
        block = own[0] + nc[0] * (own[1] + nc[1] * own[2])
        N = len(q)
        ids = torch.arange(N, device="cuda")
        out = []
        for col in range(8):
            sel = torch.nonzero(colour == col)[:, 0]
            # each particle's block in this colour, and its rank by id there
            o = [(cell[:, k] - ((col >> k) & 1)) % nc[k] // 2 * 2 + ((col >> k) & 1) for k in range(3)]
            o = [v % nc[k] for k, v in enumerate(o)]
            pb = o[0] + nc[0] * (o[1] + nc[1] * o[2])
            order = torch.argsort(pb * N + ids)
            first = torch.searchsorted(pb[order], pb[order])
            rank = torch.empty_like(ids)
            rank[order] = ids - first
            ri, rj = rank[i[sel]], rank[j[sel]]
            key = (block[sel] * N + (rj - ri)) * N + ri
            sel = sel[torch.argsort(key)]
            b = block[sel]
            start = torch.searchsorted(b, b)
            pos = torch.arange(len(sel), device="cuda") - start
            # dependency levels, all blocks side by side along their lists
            by_pos = torch.argsort(pos, stable=True)
            bounds = torch.searchsorted(pos[by_pos], torch.arange(int(pos.max()) + 2, device="cuda")).tolist() if len(sel) else [0]
            free = torch.zeros(N, dtype=torch.long, device="cuda")
            level = torch.zeros(len(sel), dtype=torch.long, device="cuda")
            for a, e in zip(bounds[:-1], bounds[1:]):
                t = by_pos[a:e]
                u, v = i[sel[t]], j[sel[t]]
                lev = torch.maximum(free[u], free[v])
                level[t] = lev
                free[u] = lev + 1
                free[v] = lev + 1
            by_level = torch.argsort(level, stable=True)
            cuts = torch.searchsorted(level[by_level], torch.arange(int(level.max()) + 2, device="cuda")).tolist() if len(sel) else [0]
            out += [sel[by_level[a:e]] for a, e in zip(cuts[:-1], cuts[1:])]
        return out

    def coeffs(self, kpar, kperp, ei, ej, dt):
        Ti, Tj = ei / self.CK, ej / self.CK
        s = Ti * Tj / (Ti + Tj)
        omd = 1.0 - s / (Ti + Tj) * 2.0 / self.CK
        mpar, mperp = torch.expm1(-2.0 * kpar * omd * dt), torch.expm1(-2.0 * kperp * omd * dt)
        s = 4.0 * s / omd
        return mpar, mperp, torch.sqrt(-s * mpar * (2.0 + mpar)), torch.sqrt(-s * mperp * (2.0 + mperp))

    def sweep(self, q, p, eps, dt, ij, rho, levels):
        p, eps = p.clone(), eps.clone()
        d = self.disp(q, ij)
        r = self.dist(d)
        unit, base = d / r[:, None], self.F(r, self.h) / (rho[ij[0]] * rho[ij[1]])
        G, U = self.randoms(ij[0], ij[1])
        scheme = self.case["scheme"]
        for t in levels:
            i, j = ij[0][t], ij[1][t]
            e, g, kpar = unit[t], G[t], 10.0 / 3.0 * base[t]
            kperp = 0.5 * kpar
            pi, pj, ei, ej = p[i], p[j], eps[i], eps[j]
            v = pi - pj
            mpar, mperp, zpar, zperp = self.coeffs(kpar, kperp, ei, ej, dt)
            vp, gp = (e * v).sum(1), (e * g).sum(1)
            dv = mperp[:, None] * v + zperp[:, None] * g + ((mpar - mperp) * vp + (zpar - zperp) * gp)[:, None] * e
            ni, nj = pi + 0.5 * dv, pj - 0.5 * dv
            de = -0.25 * ((ni - pi) * (ni + pi) + (nj - pj) * (nj + pj)).sum(1)
            ok = torch.minimum(ei, ej) + de > 0.0
            if scheme == "ssa":
                ok = torch.ones_like(ok)
            elif scheme == "ems":
                rpar, rperp, ypar, yperp = self.coeffs(kpar, kperp, ei + de, ej + de, dt)
                # reverse noise along and across e
                bpar = (-(mpar + rpar + mpar * rpar) * vp - (1 + rpar) * zpar * gp) / ypar
                vt, gt = v - vp[:, None] * e, g - gp[:, None] * e
                bt = (-(mperp + rperp + mperp * rperp)[:, None] * vt - ((1 + rperp) * zperp)[:, None] * gt) / yperp[:, None]
                a = 0.5 * ((g * g).sum(1) - bpar * bpar - (bt * bt).sum(1)) + torch.log(zpar * zperp ** 2 / (ypar * yperp ** 2))
                a = a + (self.CK - 1.0) * torch.log1p(de * (ei + ej + de) / (ei * ej))
                ok = ok & (torch.log(U[t]) <= a)
            ok = ok | ~(base[t] > 0.0)
            de = torch.where(ok & (base[t] > 0.0), de, torch.zeros_like(de))
            dp = torch.where((ok & (base[t] > 0.0))[:, None], 0.5 * dv, torch.zeros_like(dv))
            p[i] += dp
            p[j] -= dp
            eps[i] += de
            eps[j] += de
            self.n_reject += (~ok).sum()
        self.n_pairs += ij.shape[1]
        self.sweeps += 1
        return p, eps

    def steps(self, q, p, eps, dt, n, theta=1, th=None):
        """n full steps; with th given, differentiable (sweeps' increments fixed)."""
        diff = th is not None
        th = th if diff else (self.h, self.cr, self.CK)
        ij = None
        for k in range(1, n + 1):
            q, p, eps, ij = self.verlet(q, p, eps, dt, th, ij)
            if self.case["scheme"] != "none" and k % theta == 0:
                with torch.no_grad():
                    q0, p0, e0 = q.detach(), p.detach(), eps.detach()
                    rho = self.density(q0, ij, self.h)
                    p1, e1 = self.sweep(q0, p0, e0, theta * dt, ij, rho, self.schedule(q0, ij))
                p, eps = p + (p1 - p0), eps + (e1 - e0)
        return q, p, eps, ij


def exact(case, seed):
    kind = case["kind"]
    # a sweep costs about a second here whatever the size; the pair search is
    # quadratic
    sweeps = 0 if case["scheme"] == "none" else case["steps"] // (1 if kind == "fd" else case["theta"])
    searches = 1 if kind == "fd" else case["steps"] + 1
    if kind == "ensemble" or sweeps > 8 or _count(case) > 300000 or searches * _count(case) ** 2 > 2.5e11:
        return None
    if kind == "gradient" and _count(case) * case["steps"] > 70000:
        return None
    ref = _Ref(case, _box(case), seed & 0xFFFFFF)
    q, p, e = (torch.as_tensor(a, device="cuda") for a in _state(case, seed))
    q = q - ref.L * torch.floor(q / ref.L)
    dt, n = case["dt"], case["steps"]
    if kind == "gradient":
        x = [t.clone().requires_grad_() for t in (q, p, e)]
        th = torch.tensor([2.5, ref.cr, ref.CK], dtype=torch.float64, device="cuda", requires_grad=True)
        qn, pn, en, ij = ref.steps(*x, dt, n, th=th)
        rho = ref.density(qn, ij, th[0])
        _, d, f = ref.force(qn, rho, en, ij, th)
        loss = ((pn * pn).sum() + (d * f).sum()) / (3.0 * float(torch.prod(ref.L)))
        loss.backward()
        return {"loss": loss.detach(), "gq": x[0].grad, "gp": x[1].grad, "geps": x[2].grad, "gtheta": th.grad.cpu()}
    if kind == "fd":
        ij = ref.pairs(q)
        rho, levels = ref.density(q, ij, ref.h), ref.schedule(q, ij)
        for _ in range(n):
            p, e = ref.sweep(q, p, e, dt, ij, rho, levels)
        return {"p": p, "eps": e, "counts": None}
    q, p, e, _ = ref.steps(q, p, e, dt, n, theta=case["theta"])
    if kind == "host":
        return {"q": q, "p": p, "eps": e, "status": None}
    kin = 0.5 * float((p * p).sum())
    return {"q": q, "p": p, "eps": e, "E": float(e.sum()) + kin, "T_kin": 2.0 * kin / (3.0 * (len(q) - 1)),
            "T_int": float(e.mean()) / ref.CK, "n_pairs": None, "n_reject": None}
