"""The workloads that the framework's performance is followed on.

Each case is one call (or the short sequence of calls) that a user's program
repeats: a load increment of a batch of r-cells, an FE step, a relaxation, an
optimiser step, a prediction.  ``listed()`` names them, ``draw`` gives further
sizes of the same ranges, ``prepare`` makes the inputs from a seed, ``run`` is
one pass through the public entry points, ``work`` its algorithmic bytes and
operations, ``exact`` the same results in plain 64-bit torch.

MD increments here have fewer steps than production ones (400 to 1000): two
64-bit-identical starts stay comparable over tens of steps only, and one
deformation plus a few list rebuilds is the mix of the long run.  The r-cell
engine computes in FP32, so its stresses are handed on as FP32, as the
surrogate's training data are.
"""
import functools
import math

import numpy as np
import torch

from paper_1902_09171_gb300 import inputs, rcell
from paper_1902_09171_gb300 import surrogate as S

KT_CU = 300 * inputs.KB_EV
M_CU, A_CU = 63.546, 3.615
CHAIN, RHO_KG = 50, 0.85
N_MEMBERS = 4
DEV = torch.device("cuda")
EV, AMU = 1.602176634e-19, 1.66053906660e-27


def listed():
    return [
        # one quadrature point of the plain method: a 256-atom LJ copper cell, host arrays in and out
        {"name": "lj_point", "kind": "md", "pot": "lj", "cells": 1, "edge": 4, "steps": 100, "avg": 50, "skin": 0.5,
         "lanes": 1, "active": 1, "host": True},
        # the copper bar: one load increment of an 8 x 2 x 2 mesh with a 4000-atom Sutton-Chen cell per element
        {"name": "cu_bar", "kind": "fe", "pot": "sc", "mesh": "8,2,2", "edge": 10, "steps": 100, "avg": 50,
         "skin": 1.5, "lanes": 1},
        # the MD fallback of the surrogate on that bar: three of its points run MD, the others stay frozen
        {"name": "cu_fallback", "kind": "md", "pot": "sc", "cells": 32, "edge": 10, "steps": 100, "avg": 50,
         "skin": 1.5, "lanes": 1, "active": 3, "host": False},
        # the periodic-box tensile run: 32 Kremer-Grest cells at T = 0.1, chunks of 50 steps that all sample
        {"name": "kg_tensile", "kind": "md", "pot": "kg", "cells": 32, "chains": 100, "copies": 1, "steps": 50,
         "avg": 50, "skin": 0.3, "lanes": 1, "active": 32, "host": True, "kT": 0.1},
        # the polymer bar: 64 uneven cells of 5000 to 20000 beads at the autotuner's choice (lean walk, skin 0.5)
        {"name": "kg_bar", "kind": "md", "pot": "kg", "cells": 64, "chains": 0, "copies": 0, "steps": 100, "avg": 50,
         "skin": 0.5, "lanes": 0, "active": 64, "host": False, "kT": 0.3},
        # the necking bar at full size: 512 cells of 20000 beads, autotuned (lean walk, skin 0.4), one FE step
        {"name": "necking_bar", "kind": "fe", "pot": "kg", "mesh": "32,4,4", "chains": 100, "copies": 4, "steps": 40,
         "avg": 20, "skin": 0.4, "lanes": 0},
        # the statics route: FIRE on 32 glass cells after a load increment, then the pair-sum stress
        {"name": "kg_relax", "kind": "relax", "cells": 32, "chains": 100, "copies": 1, "iters": 96, "skin": 0.3},
        # surrogate training at its production shape: two AdamW steps of the ensemble, parameters read back
        {"name": "train_step", "kind": "train", "batch": 4096, "increments": 60, "updates": 2},
        # loss and gradient of one member on a small, odd batch of shorter histories
        {"name": "gradient", "kind": "gradient", "batch": 777, "increments": 25},
        # the trained ensemble on whole histories (held-out error, spread statistics)
        {"name": "predict", "kind": "predict", "batch": 4096, "increments": 60},
        # one increment of every quadrature point of the necking bar: features and the recurrent step
        {"name": "point_step", "kind": "point", "points": 512},
        # one surrogate-driven FE step of the copper bar with no point on MD
        {"name": "surrogate_fe", "kind": "surrogate_fe", "mesh": "8,2,2", "edge": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lj", "sc", "kg", "kg_fe", "relax", "train", "gradient", "predict", "point", "surrogate_fe"])
    if kind == "lj":
        n = _log(rng, 1, 32)
        return {"kind": "md", "pot": "lj", "cells": n, "edge": rng.randint(4, 9), "steps": rng.randint(40, 100),
                "avg": rng.randint(20, 40), "skin": rng.choice([0.5, 1.0]), "lanes": rng.choice([1, 2]),
                "active": n, "host": rng.random() < 0.5}
    if kind == "sc":
        n = _log(rng, 2, 48)
        return {"kind": "md", "pot": "sc", "cells": n, "edge": rng.randint(6, 11), "steps": rng.randint(20, 50),
                "avg": rng.randint(10, 20), "skin": rng.choice([1.0, 1.5]), "lanes": rng.choice([0, 1, 1, 1, 2]),
                "active": max(1, int(n * rng.choice([0.1, 1.0, 1.0]))), "host": False}
    if kind == "kg":
        n = _log(rng, 4, 96)
        return {"kind": "md", "pot": "kg", "cells": n, "chains": rng.randint(41, 130), "copies": rng.choice([1, 1, 2, 4]),
                "steps": rng.randint(30, 60), "avg": rng.randint(10, 30), "skin": rng.choice([0.3, 0.4, 0.5, 0.6]),
                "lanes": rng.choice([0, 0, 1, 2]), "active": n, "host": rng.random() < 0.3,
                "kT": rng.choice([0.1, 0.3])}
    if kind == "kg_fe":
        return {"kind": "fe", "pot": "kg", "mesh": "%d,%d,%d" % (rng.randint(4, 12), rng.randint(1, 4), rng.randint(2, 4)),
                "chains": rng.randint(60, 110), "copies": rng.choice([1, 2, 4]), "steps": rng.randint(20, 40),
                "avg": rng.randint(5, 20), "skin": rng.choice([0.4, 0.5]), "lanes": 0}
    if kind == "relax":
        return {"kind": "relax", "cells": _log(rng, 2, 48), "chains": rng.randint(41, 120), "copies": rng.choice([1, 2]),
                "iters": 32 * rng.randint(1, 3), "skin": rng.choice([0.3, 0.4])}
    if kind == "train":
        return {"kind": "train", "batch": _log(rng, 200, 4096), "increments": rng.randint(16, 60), "updates": 2}
    if kind in ("gradient", "predict"):
        return {"kind": kind, "batch": _log(rng, 20, 4096), "increments": rng.randint(8, 60)}
    if kind == "point":
        return {"kind": "point", "points": _log(rng, 8, 4096)}
    return {"kind": "surrogate_fe", "mesh": "%d,%d,%d" % (rng.randint(2, 16), rng.randint(1, 4), rng.randint(1, 4)),
            "edge": rng.randint(6, 8)}


# ---------------------------------------------------------------------------
# plain 64-bit molecular dynamics in torch: it makes the polymer melts (the
# same ones whatever the framework's code) and the exact results
# ---------------------------------------------------------------------------

class Plain:
    """A batch of cells as one flat array of atoms (`cell` says whose), with the potential of rcell_params."""

    def __init__(self, prm, x, v, H, cell, tag, chain=0):
        self.p, self.x, self.v, self.H, self.cell, self.tag = prm, x, v, H, cell, tag
        self.Hi = _inv(H)
        self.n = torch.bincount(cell, minlength=H.shape[0])
        self.first = torch.cumsum(self.n, 0) - self.n
        me = torch.arange(len(x), device=x.device)
        self.side = []
        if chain:
            self.side = [(torch.where(tag % chain > 0, me - 1, me)), torch.where(tag % chain < chain - 1, me + 1, me)]

    def apart(self, i, j, x):
        """Minimum-image x_j - x_i, i broadcastable against j; boxes are upper triangular."""
        d = x[j] - x[i]
        H, G = self.H[self.cell[i]], self.Hi[self.cell[i]]
        a, b, c = d.unbind(-1)
        na = (G[..., 0, 0] * a + G[..., 0, 1] * b + G[..., 0, 2] * c).round()
        nb = (G[..., 1, 1] * b + G[..., 1, 2] * c).round()
        nc = (G[..., 2, 2] * c).round()
        return torch.stack([a - (H[..., 0, 0] * na + H[..., 0, 1] * nb + H[..., 0, 2] * nc),
                            b - (H[..., 1, 1] * nb + H[..., 1, 2] * nc), c - H[..., 2, 2] * nc], -1)

    def build(self, reach):
        """Table of the neighbours within `reach` (rows padded with the atom itself), chain neighbours left out."""
        self.reach = reach
        rows, width = [], 1
        x = self.x.to(torch.float32)
        for c in range(len(self.n)):
            n, a = int(self.n[c]), int(self.first[c])
            xc, H, Hi = x[a:a + n], self.H[c].float(), self.Hi[c].float()
            for k in range(0, n, 2500):
                d = xc[None, :, :] - xc[k:k + 2500, None, :]
                d = d - (d @ Hi.T).round() @ H.T
                near = (d * d).sum(-1) < reach * reach
                i, j = torch.nonzero(near, as_tuple=True)
                keep = j != i + k
                rows.append((i[keep] + a + k, j[keep] + a))
        i, j = torch.cat([r[0] for r in rows]), torch.cat([r[1] for r in rows])
        for side in self.side:
            keep = side[i] != j
            i, j = i[keep], j[keep]
        count = torch.bincount(i, minlength=len(x))
        width = max(1, int(count.max()))
        place = torch.arange(len(i), device=i.device) - (torch.cumsum(count, 0) - count)[i]
        self.nb = torch.arange(len(x), device=x.device)[:, None].repeat(1, width)
        self.nb[i, place] = j

    def pairs(self, a, b):
        j = self.nb[a:b]
        me = torch.arange(a, a + len(j), device=self.x.device)[:, None]
        d = self.apart(me, j, self.x)
        r2 = (d * d).sum(-1)
        on = (j != me) & (r2 < self.p.rc ** 2)
        return d, torch.where(on, r2, torch.ones_like(r2)), on, j

    def forces(self, virial=False, floor=0.0, soft=0.0):
        """Forces and, per atom, half of its pairs' -dU/dr d (x) d / r (each pair is seen from both ends).  For melts
        in the making: squared distances no smaller than `floor`, a cosine repulsion of that height (`soft`) for LJ."""
        p, N = self.p, len(self.x)
        f = torch.zeros_like(self.x)
        W = torch.zeros(N, 3, 3, dtype=self.x.dtype, device=self.x.device) if virial else None
        step = max(1, 60_000_000 // self.nb.shape[1])
        inv = None
        if p.potential == rcell.RC_POT_SC:
            inv = torch.empty(N, dtype=self.x.dtype, device=self.x.device)
            for a in range(0, N, step):
                d, r2, on, j = self.pairs(a, a + step)
                inv[a:a + step] = ((p.sigma ** 2 / r2) ** (p.m / 2) * on).sum(1) ** -0.5
        for a in range(0, N, step):
            d, r2, on, j = self.pairs(a, a + step)
            r2 = r2.clamp_min(floor) if floor else r2
            if soft:
                r = r2.sqrt()
                g = -soft * math.pi / 1.122 * torch.sin(math.pi / 1.122 * r.clamp_max(1.122)) / r
            elif inv is None:
                s6 = (p.sigma ** 2 / r2) ** 3
                g = -24 * p.eps * s6 * (2 * s6 - 1) / r2
            else:
                q = p.sigma ** 2 / r2
                g = p.eps / r2 * (p.c * p.m / 2 * (inv[a:a + step, None] + inv[j]) * q ** (p.m / 2) - p.n * q ** (p.n / 2))
            g = g * on
            f[a:a + step] = (g[..., None] * d).sum(1)
            if virial:
                W[a:a + step] = -0.5 * torch.einsum("nk,nka,nkb->nab", g, d, d)
        me = torch.arange(N, device=self.x.device)
        for side in self.side:
            d = self.apart(me, side, self.x)
            bound = (side != me).to(d.dtype)
            r2 = torch.where(side != me, (d * d).sum(-1), torch.ones_like(bound))
            r2 = r2.clamp(floor, 0.9 * p.R0 ** 2) if floor else r2
            s6 = (p.sigma ** 2 / r2) ** 3
            wca = r2 < 2 ** (1 / 3) * p.sigma ** 2
            g = bound * (p.k_fene / (1 - r2 / p.R0 ** 2) - wca * 24 * p.eps * s6 * (2 * s6 - 1) / r2)
            f += g[:, None] * d
            if virial:
                W += -0.5 * torch.einsum("n,na,nb->nab", g, d, d)
        return f, W

    def per_cell(self, w):
        return torch.stack([w[int(a):int(a) + int(n)].sum(0) for a, n in zip(self.first, self.n)])

    def units(self):
        metal = self.p.units == rcell.RC_UNITS_METAL
        return (EV / (1e-10 * AMU) / 1e14, EV / 1e-30 / 1e9) if metal else (1.0, 1.0)

    def normals(self, step):
        """Three standard normals per atom: Philox4x32-10 of (tag, cell, evaluation) and the seed, Box-Muller."""
        low, seed = 0xFFFFFFFF, int(self.p.seed)
        c = [self.tag, self.cell_id, torch.full_like(self.tag, step & low), torch.zeros_like(self.tag)]
        k0, k1 = seed & low, seed >> 32
        for _ in range(10):
            a, b = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
            c = [((b >> 32) & low) ^ c[1] ^ k0, b & low, ((a >> 32) & low) ^ c[3] ^ k1, a & low]
            k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
        u = [(w.double() + 0.5) * 2.0 ** -32 for w in c]
        r0, r1 = (-2 * u[0].log()).sqrt(), (-2 * u[2].log()).sqrt()
        return torch.stack([r0 * (2 * math.pi * u[1]).cos(), r0 * (2 * math.pi * u[1]).sin(),
                            r1 * (2 * math.pi * u[3]).cos()], 1)

    def run(self, steps, avg):
        """steps of velocity Verlet with the force-form Langevin thermostat; mean MD-frame stress of the last avg."""
        p = self.p
        ftm, pconv = self.units()
        amp = math.sqrt(2 * p.kT * ftm / (p.mass * p.tau * p.dt))
        vol = _det(self.H)[:, None, None]
        total = torch.zeros(len(self.n), 3, 3, dtype=torch.float64, device=self.x.device)
        for s in range(steps + 1):
            if s % 50 == 49:
                self.build(self.reach)
            sample = s > steps - avg
            f, W = self.forces(virial=sample)
            a = f * (ftm / p.mass) - self.v / p.tau + amp * self.normals(s)
            if s > 0:
                self.v = self.v + 0.5 * p.dt * a
            if sample:
                K = p.mass / ftm * self.v[:, :, None] * self.v[:, None, :]
                total -= self.per_cell(K + W) * pconv / vol / avg
            if s < steps:
                self.v = self.v + 0.5 * p.dt * a
                self.x = self.x + p.dt * self.v
        return total


@functools.lru_cache(maxsize=24)
def _melt(chains, number):
    """A Kremer-Grest glass of `chains` chains at density 0.85 and about T = 0.3: random walks whose overlaps a growing
    soft repulsion pushes apart, then displacement-limited Langevin dynamics.  Returns positions (chains unwrapped) and the box edge."""
    rng = np.random.default_rng(1000 * chains + number)
    n = chains * CHAIN
    L = (n / RHO_KG) ** (1 / 3)
    step = rng.standard_normal((chains, CHAIN, 3))
    step /= np.linalg.norm(step, axis=2, keepdims=True)
    for k in range(2, CHAIN):  # no folding back
        back = np.linalg.norm(step[:, k] + step[:, k - 1], axis=1) < 1.05
        step[back, k] *= -1
    step *= 0.97
    step[:, 0] = rng.uniform(0, L, (chains, 3))
    dev = DEV
    x = torch.tensor(np.cumsum(step, 1).reshape(n, 3), device=dev)
    noise = torch.Generator(device=dev).manual_seed(77 + 1000 * chains + number)
    prm = rcell.params_kg()
    sim = Plain(prm, x, torch.zeros_like(x), L * torch.eye(3, dtype=x.dtype, device=dev)[None],
                torch.zeros(n, dtype=torch.int64, device=dev), torch.arange(n, device=dev), CHAIN)
    for kT, tau, steps, cap, top in ((1.0, 0.5, 400, 0.04, 60.0), (1.0, 0.5, 150, 0.02, 0.0), (0.3, 0.5, 250, 0.05, 0.0)):
        amp = math.sqrt(2 * kT / (tau * prm.dt))
        for k in range(steps):
            if k % 10 == 0:
                sim.build(2.0 if top else 3.1)
            f, _ = sim.forces(floor=0.5 if cap < 0.05 else 0.0, soft=2.0 + top * k / steps if top else 0.0)
            a = f - sim.v / tau + amp * torch.randn(n, 3, dtype=x.dtype, device=dev, generator=noise)
            v = sim.v + prm.dt * a
            size = prm.dt * (v * v).sum(1, keepdim=True).sqrt().clamp_min(1e-30)
            sim.v = v * (cap / size).clamp_max(1.0)
            sim.x = sim.x + prm.dt * sim.v
    return sim.x.cpu().numpy(), L


@functools.lru_cache(maxsize=24)
def _bonds(chains):
    k = np.arange(chains * CHAIN, dtype=np.int32)
    k = k[k % CHAIN < CHAIN - 1]
    return np.stack([k, k + 1], 1)


COPIES = {1: (1, 1, 1), 2: (2, 1, 1), 4: (2, 2, 1)}
UNEVEN = ((100, 1), (142, 1), (54, 2), (100, 2), (71, 4), (142, 2), (100, 4))  # (chains, copies): 5000 to 20000 beads


def _kg_cells(n, chains, copies, kT, seed):
    """n cells, each a glass repeated `copies` times, shifted by a seeded vector, with Maxwell velocities of its own."""
    rng = np.random.default_rng(seed)
    out = []
    for c in range(n):
        ch, m = UNEVEN[c % len(UNEVEN)] if chains == 0 else (chains, copies)
        x, L = _melt(ch, c % 2)
        rep = COPIES[m]
        box = np.array([L * r for r in rep])
        tiles = [x + L * np.array([i, j, k]) for i in range(rep[0]) for j in range(rep[1]) for k in range(rep[2])]
        x = np.mod(np.concatenate(tiles) + rng.uniform(0, L, 3), box)
        v = rng.standard_normal(x.shape, dtype=np.float32) * np.float32(math.sqrt(kT))
        out.append(dict(H0=np.diag(box), x0=inputs.to_f32(x), v0=inputs.to_f32(v - v.mean(0)), bonds=_bonds(ch * m)))
    return out


def _cu_cells(n, edge, seed):
    x, H = inputs.fcc(edge, edge, edge, A_CU)
    rng = np.random.default_rng(seed)
    out = []
    for c in range(n):
        s = int(rng.integers(1 << 30))
        # half of the thermal energy already in the displacements
        xc = np.mod(x + 0.06 * np.random.default_rng(s).standard_normal(x.shape) + rng.uniform(0, A_CU, 3), H[0, 0])
        out.append(dict(H0=H, x0=inputs.to_f32(xc), v0=inputs.to_f32(inputs.maxwell(len(x), M_CU, KT_CU, 0, s + 1))))
    return out


def _cells(case, n, seed):
    if case.get("pot", "kg") == "kg":
        return _kg_cells(n, case["chains"], case["copies"], case.get("kT", 0.3), seed)
    return _cu_cells(n, case["edge"], seed)


def _params(case, seed):
    pot = case.get("pot", "kg")
    if pot == "lj":
        return rcell.params_lj_cu(kT=KT_CU, seed=seed % 1000 + 1, skin=case["skin"])
    if pot == "sc":
        return rcell.params_sc_cu(kT=KT_CU, seed=seed % 1000 + 1, skin=case["skin"])
    return rcell.params_kg(kT=case.get("kT", 0.3), seed=seed % 1000 + 1, skin=case["skin"])


def _level(k):
    """Load levels 1, 2 .. 6, 5 .. 0, 1 ..: cyclic loading, so that a pass can be repeated for ever."""
    return 6 - abs((k + 1) % 12 - 6)


def _paths(case, n, seed):
    """F of every cell at load levels 0 .. 6: stretch with lateral contraction, and a little shear."""
    rng = np.random.default_rng(seed + 5)
    de = 0.0025 if case.get("pot", "kg") == "kg" else 0.002
    G = np.zeros((n, 3, 3))
    G[:, 0, 0] = de * rng.uniform(0.6, 1.0, n)
    G[:, 1, 1] = G[:, 2, 2] = -0.35 * G[:, 0, 0]
    G += 0.1 * de * rng.uniform(-1, 1, G.shape)
    return np.eye(3) + np.arange(7)[:, None, None, None] * G


class State:
    """A user's program between two calls: contexts, buffers, and how far the loading has come."""

    def __init__(self):
        self.k, self.undo = 0, []

    def __del__(self):
        for free, handle in self.undo:
            free(handle)


@functools.lru_cache(maxsize=1)
def _stream():
    return torch.cuda.Stream()


def _zeros(*shape, dtype=torch.float64):
    return torch.zeros(shape, dtype=dtype, device=DEV)


def _theta(seed, members, spread):
    """Parameter vectors of an ensemble: uniform +-1/sqrt(fan_in) weights, small biases; `spread` > 0: members that
    differ from the first by that share, as members trained on the same data do."""
    rng = np.random.default_rng(seed)

    def one():
        parts = []
        for k, n, kl, nl in ((144, 256, 143, 256), (256, 256, 256, 256), (256, 256, 256, 256), (256, 144, 256, 134)):
            w = np.zeros((k, n))
            w[:kl, :nl] = rng.uniform(-1, 1, (kl, nl)) / math.sqrt(k)
            b = np.zeros(n)
            b[:nl] = 0.05 * rng.standard_normal(nl)
            parts += [w.ravel(), b]
        return np.concatenate(parts)

    first = one()
    rest = [one() if not spread else first + spread * one() for _ in range(members - 1)]
    return [t.astype(np.float32) for t in [first] + rest]


def _surrogate(s, seed, batch, increments, spread, u_scale, s_scale):
    st = _stream()
    s.sur = S.sur_create(N_MEMBERS, batch, increments, seed % 1000, stream=st)
    s.undo.append((S.sur_destroy, s.sur))
    S.sur_set_scaling(s.sur, u_scale, s_scale)
    s.theta = _theta(seed, N_MEMBERS, spread)
    for m in range(N_MEMBERS):
        S.sur_set_params(s.sur, m, s.theta[m])


def _histories(seed, batch, increments):
    """Smooth strain-like histories and stresses that depend on them."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    U = torch.randn(batch, increments, 15, device=DEV, generator=g)
    ramp = torch.linspace(0.1, 1.0, increments, device=DEV)[None, :, None]
    U[:, :, 9:] = ramp * torch.randn(batch, 1, 6, device=DEV, generator=g) + 0.1 * U[:, :, 9:]
    Y = U[:, :, 9:] - 0.3 * U[:, :, 9:] ** 2 + 0.2 * torch.randn(batch, increments, 6, device=DEV, generator=g)
    return U.contiguous(), Y.contiguous()


def _points(seed, n):
    """Deformations of n quadrature points at load levels 0 .. 6, and their recurrent states."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    F, dF = (torch.randn(n, 3, 3, dtype=torch.float64, device=DEV, generator=g) for _ in range(2))
    F = torch.eye(3, dtype=torch.float64, device=DEV) + 0.03 * F
    h = torch.tanh(0.3 * torch.randn(N_MEMBERS, n, 128, device=DEV, generator=g))
    return [F + 0.004 * k * dF for k in range(7)], h


SCALES = (np.array([0.02] * 9 + [0.03] * 6, np.float32), np.full(6, 1.5, np.float32))


def _bar(case, seed):
    """Mesh, boundary conditions and FE parameters of the copper bar and the necking bar."""
    n = tuple(int(v) for v in case["mesh"].split(","))
    if case.get("pot", "sc") == "kg":
        h = (case["chains"] * CHAIN * case["copies"] / RHO_KG) ** (1 / 3)
        X, conn = inputs.necking_mesh(*n, h)
        prm = (RHO_KG, 2.0, 1.0, 1.0)
    else:
        h = case["edge"] * A_CU
        X, conn = inputs.hex_mesh(*n, n[0] * h, n[1] * h, n[2] * h)
        rho = 4 * M_CU / A_CU ** 3 / 60.2214
        dt = 0.5 * h / math.sqrt(130.0 / rho)
        prm = (rho, dt, 2.0 / dt, 6.5)
    mask, val = inputs.uniaxial_bc(X, n[0] * h)
    return X, conn, mask, val, prm


def _make_bar(s, case, seed):
    X, conn, mask, val, prm = _bar(case, seed)
    s.fe = rcell.fe_create(X, conn, mask, val, *prm, stream=_stream())
    s.undo.append((rcell.fe_destroy, s.fe))
    g = np.zeros_like(X)
    g[:, 0] = X[:, 0]
    rcell.fe_set_predictor(s.fe, g)
    s.ne = len(conn)
    s.dl = 0.002 * (1 + 0.01 * (seed % 50))  # strain of one load level


def prepare(case, seed):
    rcell.load()
    st, kind = _stream(), case["kind"]
    s = State()
    s.case = case
    with torch.cuda.stream(st):
        if kind in ("md", "relax"):
            n = case["cells"]
            s.rc = rcell.rcell_create(_params(case, seed), _cells(case, n, seed), stream=st)
            s.undo.append((rcell.rcell_destroy, s.rc))
            paths = _paths(case, n, seed)
            s.F = list(paths) if case.get("host", True) else [torch.tensor(F, device=DEV) for F in paths]
            if kind == "md":
                rcell.rcell_set_tuning(s.rc, case["lanes"], 1)
                if case["active"] < n:
                    on = np.zeros(n, np.int32)
                    on[np.random.default_rng(seed + 9).permutation(n)[:case["active"]]] = 1
                    rcell.rcell_set_active(s.rc, on)
                    s.on = torch.tensor(np.nonzero(on)[0], device=DEV)
        elif kind == "fe":
            _make_bar(s, case, seed)
            s.rc = rcell.rcell_create(_params(case, seed), _cells(case, s.ne, seed), stream=st)
            s.undo.append((rcell.rcell_destroy, s.rc))
            rcell.rcell_set_tuning(s.rc, case["lanes"], 1)
        elif kind in ("train", "gradient", "predict"):
            B, T = case["batch"], case["increments"]
            one = np.ones(15, np.float32), np.ones(6, np.float32)
            _surrogate(s, seed, B, T, 0.0, *one)
            s.data = [_histories(seed + 31 * k, B, T) for k in range(3 if kind == "train" else 1)]
            if kind == "train":  # mid-training: the optimiser's moments are filled (a warm-up at learning rate 0)
                for U, Y in s.data:
                    S.sur_train_step(s.sur, U, Y, 0.0, n_members=N_MEMBERS, want_loss=False)
        elif kind == "point":
            n = case["points"]
            _surrogate(s, seed, n, 1, 0.05, *SCALES)
            s.F, s.h = _points(seed, n)
            s.u, s.mean, s.spread = (_zeros(n, k, dtype=torch.float32) for k in (15, 6, 1))
        else:
            _make_bar(s, case, seed)
            s.rc = rcell.rcell_create(_params({"pot": "sc", "skin": 1.5}, seed), _cu_cells(s.ne, case["edge"], seed), stream=st)
            s.undo.append((rcell.rcell_destroy, s.rc))
            _surrogate(s, seed, s.ne, 1, 0.02, SCALES[0], SCALES[1] * 0.02)
            s.h = _zeros(N_MEMBERS, s.ne, 128, dtype=torch.float32)
            s.Fp = torch.eye(3, dtype=torch.float64, device=DEV).repeat(s.ne, 1, 1)
            s.flag, s.spread = _zeros(s.ne, dtype=torch.int32), _zeros(s.ne, dtype=torch.float32)
    torch.cuda.synchronize()
    return s


def run(s):
    with torch.cuda.stream(_stream()):
        return _pass(s, s.case, s.case["kind"])


def _pass(s, c, kind):
    level = _level(s.k)
    s.k += 1
    if kind == "md":
        rcell.rcell_set_deformation(s.rc, s.F[level])
        rcell.rcell_run(s.rc, c["steps"], c["avg"])
        if c["host"]:
            return [v.astype(np.float32) for v in rcell.rcell_stress(s.rc)]
        sig, se, P = (_zeros(c["cells"], *k) for k in ((6,), (6,), (3, 3)))
        rcell.rcell_stress(s.rc, sig, se, P)
        if c["active"] < c["cells"]:
            sig, se, P = sig[s.on], se[s.on], P[s.on]
        return [sig.float(), se.float(), P.float()]
    if kind == "fe":
        P, F = _zeros(s.ne, 3, 3), _zeros(s.ne, 3, 3)
        rcell.fe_step(s.fe, s.rc, s.dl * level, c["steps"], c["avg"], None)
        rcell.fe_get_P(s.fe, P)
        rcell.fe_get_F(s.fe, F)
        return [P.float(), F.float()]
    if kind == "relax":
        rcell.rcell_set_deformation(s.rc, s.F[level])
        moves = rcell.rcell_minimize(s.rc, c["iters"], 1e-2, 0.005, 0.05, 0.05)
        sig, P = _zeros(c["cells"], 6), _zeros(c["cells"], 3, 3)
        rcell.rcell_stress_static(s.rc, sig, P)
        return [sig.float(), P.float(), moves]
    if kind == "train":
        for k in range(c["updates"]):
            U, Y = s.data[k % len(s.data)]
            S.sur_train_step(s.sur, U, Y, 1e-3, n_members=N_MEMBERS, want_loss=False)
        return [S.sur_get_params(s.sur, m) for m in range(N_MEMBERS)]
    if kind == "gradient":
        loss, grad = S.sur_loss_grad(s.sur, 1, *s.data[0])
        return [np.float32(loss), grad]
    if kind == "predict":
        out = torch.empty(N_MEMBERS, c["batch"], c["increments"], 6, device=DEV)
        S.sur_predict(s.sur, s.data[0][0], out)
        return [out]
    if kind == "point":
        S.sur_features(s.F[_level(s.k - 2) if s.k > 1 else 0], s.F[level], s.u, stream=_stream())
        S.sur_step(s.sur, s.u, s.h, 0.5, s.mean, s.spread)
        return [s.mean, s.spread, s.h]
    rcell.fe_step_surrogate(s.fe, s.rc, s.sur, s.dl * level, 50, 25, 0.02, 0.01, 0.02, False, s.h, s.Fp, s.flag, s.spread)
    P = _zeros(s.ne, 3, 3)
    rcell.fe_get_P(s.fe, P)
    return [P.float(), s.Fp.float(), s.spread, s.flag, s.h]


# ---------------------------------------------------------------------------
# algorithmic work and the 64-bit results
# ---------------------------------------------------------------------------

NET = 2 * (144 * 256 + 2 * 256 * 256 + 256 * 144)  # operations of one increment of one member
PARAMS = S.SUR_N_PARAMS


def _atoms(case):
    if case["kind"] in ("fe", "surrogate_fe"):
        n = math.prod(int(v) for v in case["mesh"].split(","))
    else:
        n = case.get("active", case.get("cells"))
    if case.get("pot", "kg") != "kg":
        return n, n * 4 * case["edge"] ** 3
    if case["chains"] == 0:
        return n, sum(CHAIN * UNEVEN[c % len(UNEVEN)][0] * UNEVEN[c % len(UNEVEN)][1] for c in range(n))
    return n, n * CHAIN * case["chains"] * case["copies"]


def work(case):
    kind = case["kind"]
    if kind in ("md", "fe", "relax"):
        cells, atoms = _atoms(case)
        pot = case.get("pot", "kg")
        # pairs inside the cutoff per atom, each once, and operations per pair, plus those of an atom (and its bond)
        pairs, per_pair, virial, per_atom = {"lj": (32.7, 38, 12, 40), "sc": (66.8, 56, 12, 40), "kg": (27.8, 26, 12, 80)}[pot]
        steps = case["iters"] if kind == "relax" else case["steps"] + 1
        avg = 1 if kind == "relax" else case["avg"]
        # positions and velocities in and out once (bond partners in), the cells' results
        return {"bytes": atoms * (48 + (8 if pot == "kg" else 0)) + cells * 400,
                "flops": atoms * (steps * (pairs * per_pair + per_atom) + avg * pairs * virial)}
    if kind == "point":
        n = case["points"]
        return {"bytes": n * (144 + 28 + N_MEMBERS * 1024) + N_MEMBERS * PARAMS * 2, "flops": n * N_MEMBERS * NET}
    if kind == "surrogate_fe":
        n = math.prod(int(v) for v in case["mesh"].split(","))
        return {"bytes": n * (500 + N_MEMBERS * 1024) + N_MEMBERS * PARAMS * 2, "flops": n * N_MEMBERS * NET}
    rows = case["batch"] * case["increments"]
    if kind == "train":
        return {"bytes": case["updates"] * (rows * 84 + N_MEMBERS * PARAMS * 24),
                "flops": case["updates"] * 3 * N_MEMBERS * rows * NET}
    if kind == "gradient":
        return {"bytes": rows * 84 + PARAMS * 8, "flops": 3 * rows * NET}
    return {"bytes": rows * (60 + 24 * N_MEMBERS) + N_MEMBERS * PARAMS * 2, "flops": N_MEMBERS * rows * NET}


def _split(F):
    """F = Q R with a positive diagonal of R."""
    Q, R = torch.linalg.qr(F.cpu())
    sign = torch.sign(torch.diagonal(R, dim1=-2, dim2=-1))
    return (Q * sign[:, None, :]).to(DEV), (sign[:, :, None] * R).to(DEV)


def _inv(A):
    return torch.linalg.inv(A.cpu()).to(DEV)


def _det(A):
    return torch.linalg.det(A.cpu()).to(DEV)


def _voigt(S9):
    return torch.stack([S9[:, 0, 0], S9[:, 1, 1], S9[:, 2, 2], S9[:, 0, 1], S9[:, 0, 2], S9[:, 1, 2]], 1)


def _plain(prm, cells, ids, F, reach):
    """The cells `ids` after the deformation F, as a Plain batch with its neighbour table."""
    Q, R = _split(F)
    H0 = torch.tensor(np.stack([c["H0"] for c in cells]), device=DEV)
    n = [len(c["x0"]) for c in cells]
    cell = torch.repeat_interleave(torch.arange(len(n), device=DEV), torch.tensor(n, device=DEV))
    x = torch.tensor(np.concatenate([c["x0"] for c in cells]), device=DEV)
    v = torch.tensor(np.concatenate([c["v0"] for c in cells]), device=DEV)
    x = torch.einsum("nab,nb->na", R[cell], x)
    tag = torch.cat([torch.arange(k, device=DEV) for k in n])
    sim = Plain(prm, x, v, R @ H0, cell, tag, CHAIN if prm.potential == rcell.RC_POT_KG else 0)
    sim.cell_id = torch.tensor(ids, device=DEV)[cell]
    sim.build(reach)
    return sim, Q


def _exact_md(case, prm, cells, ids, F):
    reach = prm.rc + (1.1 if case.get("pot", "kg") == "kg" else 1.6)
    sig, P, k = [], [], 0
    while k < len(cells):  # as many cells at a time as fit well
        m, atoms = k, 0
        while m < len(cells) and (m == k or atoms + len(cells[m]["x0"]) <= 300_000):
            atoms += len(cells[m]["x0"])
            m += 1
        sim, Q = _plain(prm, cells[k:m], ids[k:m], F[k:m], reach)
        s = Q @ sim.run(case["steps"], min(case["avg"], case["steps"])) @ Q.transpose(1, 2)
        sig.append(_voigt(s))
        P.append(_det(F[k:m])[:, None, None] * s @ _inv(F[k:m]).transpose(1, 2))
        k = m
    return torch.cat(sig), torch.cat(P)


def _exact_relax(case, prm, cells, F):
    """FIRE per cell, then P = 1/(2 V0) sum dE/dr r (x) R / r, R = H0 H^-1 r, rotated to the FE frame."""
    sim, Q = _plain(prm, cells, list(range(len(cells))), F, prm.rc + 1.1)
    n, c = len(cells), sim.cell
    one = torch.ones(n, dtype=torch.float64, device=DEV)
    dt, alpha, npos = 0.005 * one, 0.1 * one, 0 * one
    v = torch.zeros_like(sim.x)
    for it in range(case["iters"]):
        if it % 16 == 15:
            sim.build(prm.rc + 1.1)
        f, _ = sim.forces()
        p, vv, ff = (sim.per_cell((a * b).sum(1)) for a, b in ((f, v), (v, v), (f, f)))
        up = p > 0
        mixed = (1 - alpha)[c, None] * v + (alpha * (vv / ff).sqrt())[c, None] * f
        v = torch.where(up[c, None], mixed, torch.zeros_like(v))
        npos = torch.where(up, npos + 1, 0 * npos)
        fast = up & (npos > 5)
        dt = torch.where(fast, (1.1 * dt).clamp_max(0.05), torch.where(up, dt, 0.5 * dt))
        alpha = torch.where(fast, 0.99 * alpha, torch.where(up, alpha, 0.1 * one))
        v = v + dt[c, None] * f
        size = dt[c, None] * (v * v).sum(1, keepdim=True).sqrt().clamp_min(1e-300)
        v = v * (0.05 / size).clamp_max(1.0)
        sim.x = sim.x + dt[c, None] * v
    _, W = sim.forces(virial=True)
    W = sim.per_cell(W)  # -1/2 sum over ordered pairs of dE/dr d (x) d / r
    H0 = torch.tensor(np.stack([k["H0"] for k in cells]), device=DEV)
    P = Q @ (-(W @ _inv(sim.H).transpose(1, 2) @ H0.transpose(1, 2)) / _det(H0)[:, None, None])
    s = P @ F.transpose(1, 2) / _det(F)[:, None, None]
    return _voigt(0.5 * (s + s.transpose(1, 2))), P


def _net(theta, U, h):
    """Stresses (B, T, 6) and the last state of one member; U already scaled."""
    at, w = 0, []
    for k, n in ((144, 256), (256, 256), (256, 256), (256, 144)):
        w.append((theta[at:at + k * n].view(k, n), theta[at + k * n:at + k * n + n]))
        at += k * n + n
    out = []
    for t in range(U.shape[1]):
        a = torch.cat([U[:, t], h, torch.zeros_like(h[:, :1])], 1)
        for W, b in w[:3]:
            a = torch.nn.functional.gelu(a @ W + b)
        o = a @ w[3][0] + w[3][1]
        out.append(o[:, :6])
        h = torch.tanh(o[:, 6:134])
    return torch.stack(out, 1), h


def _loss_grad(theta, U, Y):
    """Loss and gradient, a part of the batch at a time."""
    theta = theta.clone().requires_grad_(True)
    total = 0.0
    for a in range(0, len(U), 1024):
        u, y = U[a:a + 1024].double(), Y[a:a + 1024].double()
        out, _ = _net(theta, u, torch.zeros(len(u), 128, dtype=torch.float64, device=DEV))
        part = ((out - y) ** 2).sum() / Y.numel()
        part.backward()
        total += float(part.detach())
    return total, theta.grad


def _features(F0, F1):
    E = 0.5 * (F1.transpose(1, 2) @ F1 - torch.eye(3, dtype=F1.dtype, device=F1.device))
    return torch.cat([(F1 - F0).reshape(-1, 9), _voigt(E)], 1)


def _ensemble(thetas, u, h, scale, floor):
    outs = [_net(t, u[:, None], h[m]) for m, t in enumerate(thetas)]
    s = torch.stack([o[0][:, 0] for o in outs]) * scale
    mean = s.mean(0)
    spread = s.var(0).sum(1).sqrt() / mean.norm(dim=1).clamp_min(floor)
    return mean, spread, torch.stack([o[1] for o in outs])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("md", "relax"):
        n = case["cells"]
        cells, prm = _cells(case, n, seed), _params(case, seed)
        F = torch.tensor(_paths(case, n, seed)[1], device=DEV)
        if kind == "relax":
            return [*_exact_relax(case, prm, cells, F), None]
        ids = sorted(np.random.default_rng(seed + 9).permutation(n)[:case["active"]].tolist())
        sig, P = _exact_md(case, prm, [cells[i] for i in ids], ids, F[ids])
        return [sig, None, P]
    if kind == "fe":
        X, conn, _, _, _ = _bar(case, seed)
        ne = len(conn)
        if ne * len(_cells(case, 1, seed)[0]["x0"]) > 4_000_000:
            return None
        F = torch.eye(3, dtype=torch.float64, device=DEV).repeat(ne, 1, 1)
        F[:, 0, 0] += 0.002 * (1 + 0.01 * (seed % 50))  # the predictor's affine field meets the boundary conditions
        _, P = _exact_md(case, _params(case, seed), _cells(case, ne, seed), list(range(ne)), F)
        return [P, None]
    thetas = lambda spread: [torch.tensor(t, dtype=torch.float64, device=DEV) for t in _theta(seed, N_MEMBERS, spread)]  # noqa: E731
    if kind in ("train", "gradient", "predict"):
        B, T = case["batch"], case["increments"]
        data = [_histories(seed + 31 * k, B, T) for k in range(3 if kind == "train" else 1)]
        if kind == "gradient":
            loss, grad = _loss_grad(thetas(0.0)[1], *data[0])
            return [loss, grad]
        if kind == "predict":
            with torch.no_grad():
                h = torch.zeros(B, 128, dtype=torch.float64, device=DEV)
                return [torch.stack([_net(t, data[0][0].double(), h)[0] for t in thetas(0.0)])]
        out = []
        for t in thetas(0.0):
            m, v = torch.zeros_like(t), torch.zeros_like(t)
            for k, (U, Y) in enumerate(data + data[:case["updates"]]):
                g = _loss_grad(t, U, Y)[1]
                m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
                if k >= len(data):
                    bias1, bias2 = 1 - 0.9 ** (k + 1), 1 - 0.999 ** (k + 1)
                    t = t - 1e-3 * ((m / bias1) / ((v / bias2).sqrt() + 1e-8) + 0.01 * t)
            out.append(t)
        return out
    with torch.no_grad():
        scale = torch.tensor(SCALES[0], dtype=torch.float64, device=DEV)
        if kind == "point":
            F, h = _points(seed, case["points"])
            mean, spread, h = _ensemble(thetas(0.05), _features(F[0], F[1]) / scale, h.double(), 1.5, 0.5)
            return [mean, spread[:, None], h]
        _, conn, _, _, _ = _bar(case, seed)
        ne = len(conn)
        one = torch.eye(3, dtype=torch.float64, device=DEV).repeat(ne, 1, 1)
        F = one.clone()
        F[:, 0, 0] += 0.002 * (1 + 0.01 * (seed % 50))
        zero = torch.zeros(N_MEMBERS, ne, 128, dtype=torch.float64, device=DEV)
        mean, spread, h = _ensemble(thetas(0.02), _features(one, F) / scale, zero, 0.03, 0.02)
        s = mean[:, [0, 3, 4, 3, 1, 5, 4, 5, 2]].view(-1, 3, 3)
        P = _det(F)[:, None, None] * s @ _inv(F).transpose(1, 2)
        return [P, F, spread, None, h]
