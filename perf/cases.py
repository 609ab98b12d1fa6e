"""What the framework is timed on: its own uses, through its public entry points.

A case is one call that a program makes again and again: an evaluation of the
exchange potential V_B with every bead force, the same through autograd, some
molecular-dynamics steps, or either of them for a batch of replicas.  Sizes
come from the repository's workloads: N = 16 and 64 trapped bosons, N = 1024
with a Gaussian repulsion, the 256-replica batch, liquid helium on FCC
lattices, and the largest system a context takes.  ``exact`` restates each in
float64 torch, with none of the repository's code.
"""
import math

import numpy as np
import torch

from paper_2305_18025_gb300.exchange import (BatchedExchangeEnergy, ExchangeEnergy, RingPolymerMD,
                                             exchange_potential)

# liquid helium in angstrom, kelvin and amu: hbar, mass, temperature, number
# density, Lennard-Jones epsilon, sigma and cutoff, and 1 fs in the time unit
HBAR, HE_M, HE_T, HE_RHO = 6.9648, 4.0026, 1.5, 0.0218
HE_LJ = (10.22, 2.556, 2.5 * 2.556)
HE_DT = 0.001 / 1.0967


def listed():
    return [
        # the smallest system of the configurations: one evaluation, all latency and launches
        {"name": "trap16_forces_fp64", "kind": "forces", "system": "trap", "N": 16, "P": 8, "beta": 2.0,
         "precision": "fp64"},
        # a differentiable energy inside a torch program: forward and backward
        {"name": "trap64_autograd_fp64", "kind": "autograd", "system": "trap", "N": 64, "P": 32, "beta": 1.0,
         "precision": "fp64"},
        # sampling of a small ideal gas in a trap, energies read every 20 steps
        {"name": "trap64_md_fp64", "kind": "md", "system": "trap", "N": 64, "P": 32, "beta": 2.0,
         "precision": "fp64", "dt": 0.005, "gauss": 0.0, "steps": 20},
        # the headline workload in the two precision forms it compares
        {"name": "trap1024_forces_mixed", "kind": "forces", "system": "trap", "N": 1024, "P": 32, "beta": 1.0,
         "precision": "mixed"},
        {"name": "trap1024_forces_fp64", "kind": "forces", "system": "trap", "N": 1024, "P": 32, "beta": 1.0,
         "precision": "fp64"},
        # ragged sizes, neighbours that overlap: long exchange cycles carry the weight
        {"name": "chain1601_forces_mixed", "kind": "forces", "system": "chain", "N": 1601, "P": 35, "beta": 1.0,
         "precision": "mixed"},
        # interacting trapped bosons, energies read every 10 (4) steps
        {"name": "trap1024_md_mixed", "kind": "md", "system": "trap", "N": 1024, "P": 32, "beta": 1.0,
         "precision": "mixed", "dt": 0.01, "gauss": 3.0, "steps": 10},
        {"name": "trap1024_md_fp64", "kind": "md", "system": "trap", "N": 1024, "P": 32, "beta": 1.0,
         "precision": "fp64", "dt": 0.01, "gauss": 3.0, "steps": 4},
        # many small systems of uneven N, P, beta at once: one evaluation, and sampling
        {"name": "replicas256_forces_mixed", "kind": "batch_forces", "system": "replicas", "R": 256, "N": 512, "sizes": 11,
         "precision": "mixed"},
        {"name": "replicas256_md_mixed", "kind": "batch_md", "system": "replicas", "R": 256, "N": 512, "sizes": 11,
         "precision": "mixed", "dt": 0.01, "gauss": 1.0, "steps": 4},
        # bulk liquid: periodic box, Lennard-Jones by cell lists
        {"name": "helium4000_md_mixed", "kind": "md", "system": "helium", "cells": 10, "N": 4000, "P": 64,
         "precision": "mixed", "dt": HE_DT, "gauss": 0.0, "steps": 5},
        # the largest N a context takes (no tables of O(N^2)), the same liquid
        {"name": "helium16384_forces_mixed", "kind": "forces", "system": "helium", "cells": 16, "N": 16384, "P": 16,
         "precision": "mixed"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forces", "forces", "forces", "autograd", "md", "md", "batch_forces", "batch_md", "helium_md",
                       "helium_forces"])
    precision = rng.choice(["fp64", "mixed"])
    beta = round(math.exp(rng.uniform(math.log(0.5), math.log(4.0))), 3)
    P = _log_int(rng, 4, 64)
    if kind in ("forces", "autograd"):
        return {"kind": kind, "system": rng.choice(["trap", "chain"]),
                "N": _log_int(rng, 12, 4096 if kind == "forces" else 1024), "P": P, "beta": beta,
                "precision": precision}
    if kind == "md":
        return {"kind": "md", "system": "trap", "N": _log_int(rng, 16, 1024), "P": P, "beta": beta,
                "precision": precision, "dt": 0.005, "gauss": rng.choice([0.0, 1.0, 3.0]), "steps": rng.randint(2, 10)}
    if kind in ("batch_forces", "batch_md"):
        c = {"kind": kind, "system": "replicas", "R": _log_int(rng, 8, 256), "N": _log_int(rng, 48, 512),
             "sizes": rng.randint(1, 10 ** 6), "precision": precision}
        if kind == "batch_md":
            c.update(dt=0.01, gauss=rng.choice([0.0, 1.0]), steps=rng.randint(2, 4))
        return c
    cells = rng.randint(3, 10) if kind == "helium_md" else rng.randint(3, 15)
    c = {"kind": "md" if kind == "helium_md" else "forces", "system": "helium", "cells": cells, "N": 4 * cells ** 3,
         "P": _log_int(rng, 8, 64 if cells <= 10 else 16), "precision": precision if cells <= 8 else "mixed"}
    if kind == "helium_md":
        c.update(dt=HE_DT, gauss=0.0, steps=rng.randint(2, 5))
    return c


# --------------------------------------------------------------- inputs
def _rng(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _box(case):
    return case["cells"] * (4.0 / HE_RHO) ** (1.0 / 3.0) if case["system"] == "helium" else 0.0


def _trap(g, N, P):
    """Centres N(0, 1) per axis, bead offsets N(0, 0.1)."""
    return _normal(g, N, 1, 3) + 0.1 * _normal(g, N, P, 3)


def _sizes(case):
    """(N, P, m, omega_P, beta) of a single system."""
    beta = 1.0 / HE_T if case["system"] == "helium" else case["beta"]
    m, hbar = (HE_M, HBAR) if case["system"] == "helium" else (1.0, 1.0)
    return case["N"], case["P"], m, math.sqrt(case["P"]) / (beta * hbar), beta


def _replicas(case):
    """Per replica N, P and beta: N ~ U[16, case N], P of 16, 32, 64, beta ~ U[0.5, 4]."""
    g = torch.Generator().manual_seed(case["sizes"])
    R = case["R"]
    N = torch.randint(16, case["N"] + 1, (R,), generator=g).tolist()
    P = [(16, 32, 64)[i] for i in torch.randint(0, 3, (R,), generator=g).tolist()]
    beta = (0.5 + 3.5 * torch.rand(R, dtype=torch.float64, generator=g)).tolist()
    return N, P, beta


def _positions(case, seed):
    g = _rng(seed)
    if case["system"] == "replicas":
        N, P, _ = _replicas(case)
        return [_trap(g, n, p) for n, p in zip(N, P)]
    N, P = case["N"], case["P"]
    if case["system"] == "trap":
        return _trap(g, N, P)
    if case["system"] == "chain":  # neighbours overlap: a random walk of centres with steps N(0, 0.05)
        return torch.cumsum(0.05 * _normal(g, N, 1, 3), 0) + 0.1 * _normal(g, N, P, 3)
    cells, a = case["cells"], _box(case) / case["cells"]
    ax = torch.arange(cells, dtype=torch.float64, device="cuda")
    grid = torch.cartesian_prod(ax, ax, ax)
    basis = torch.tensor([[0, 0, 0], [.5, .5, 0], [.5, 0, .5], [0, .5, .5]], dtype=torch.float64, device="cuda")
    centres = ((grid[:, None] + basis).reshape(-1, 3) + 0.25) * a
    return centres[:, None] + 0.05 * _normal(g, N, P, 3)


def _velocities(case, seed, pos):
    """Maxwell-Boltzmann at 1/beta."""
    g = _rng(seed + 7919)
    if isinstance(pos, list):
        return [_normal(g, *x.shape) / math.sqrt(b) for x, b in zip(pos, _replicas(case)[2])]
    _, _, m, _, beta = _sizes(case)
    return _normal(g, *pos.shape) / math.sqrt(m * beta)


def _seed_md(seed):
    return 1 + seed % 1000003


# ------------------------------------------------------------ the calls
def prepare(case, seed):
    kind, pos = case["kind"], _positions(case, seed)
    s = {"kind": kind}
    if kind in ("batch_forces", "batch_md"):
        N, P, beta = _replicas(case)
        md = None
        if kind == "batch_md":
            md = dict(dt=case["dt"], gamma=1.0, omega0=1.0, seed=_seed_md(seed),
                      gaussian=(case["gauss"], 0.5) if case["gauss"] else None)
            s["stream"] = torch.cuda.Stream()
        s["eng"] = BatchedExchangeEnergy(N, P, 1.0, [math.sqrt(p) / b for p, b in zip(P, beta)], beta,
                                         precision=case["precision"], md=md, stream=s.get("stream"))
        s["x"] = s["eng"].pack(pos)
        if kind == "batch_md":
            s["v"] = s["eng"].pack(_velocities(case, seed, pos))
            s["steps"] = case["steps"]
        return s
    N, P, m, wP, beta = _sizes(case)
    s["x"] = pos
    if kind == "md":
        s["stream"] = torch.cuda.Stream()
        helium = case["system"] == "helium"
        s["eng"] = RingPolymerMD(N, P, m, wP, beta, dt=case["dt"], gamma=1.0, omega0=0.0 if helium else 1.0,
                                 gaussian=(case["gauss"], 0.5) if case["gauss"] else None,
                                 lennard_jones=HE_LJ if helium else None, box=_box(case), seed=_seed_md(seed),
                                 precision=case["precision"], stream=s["stream"])
        s["v"] = _velocities(case, seed, pos)
        s["steps"] = case["steps"]
    else:
        s["eng"] = ExchangeEnergy(N, P, m, wP, beta, precision=case["precision"], box=_box(case))
        if kind == "autograd":
            s["x"].requires_grad_(True)
    return s


def run(s):
    kind = s["kind"]
    if kind in ("forces", "batch_forces"):
        V, F = s["eng"].forces(s["x"])
        return {"V": V, "F": F}
    if kind == "autograd":
        s["x"].grad = None
        V = exchange_potential(s["x"], s["eng"])
        V.backward()
        return {"V": V, "grad": s["x"].grad}
    energies = s["eng"].step(s["x"], s["v"], s["steps"])
    return {"x": s["x"], "v": s["v"], "energies": energies}


def work(case):
    """Bytes: positions (and velocities) read, forces (or both) written, once a
    pass.  Operations: per pair of particles a distance, a power, a step of
    each recursion, a probability and its sums (30); per bead its two springs
    (20); per pair of beads a distance and a force (20)."""
    if case["system"] == "replicas":
        n, p = case["N"] / 2 + 8, 112 / 3
        n2 = (case["N"] ** 3 - 16 ** 3) / (3 * (case["N"] - 16 + 1e-9))  # mean of N^2
        beads, pairs, bead_pairs = case["R"] * n * p, case["R"] * n2 / 2, case["R"] * n2 * p / 2
    else:
        N, P = case["N"], case["P"]
        beads, pairs, bead_pairs = N * P, N * (N + 1) / 2, N * (N - 1) / 2 * P
    if case["kind"] not in ("md", "batch_md"):
        return {"bytes": 48.0 * beads, "flops": 30.0 * pairs + 20.0 * beads}
    if case["system"] == "helium":  # partners inside the cutoff
        bead_pairs = beads / 2 * HE_RHO * 4.0 / 3.0 * math.pi * HE_LJ[2] ** 3
    elif not case["gauss"]:
        bead_pairs = 0.0
    k = case["steps"] + 1  # a step each, and the force at the start
    return {"bytes": 96.0 * beads * case["steps"], "flops": k * (30.0 * pairs + 40.0 * beads + 20.0 * bead_pairs)}


# ------------------------------------------------- the same in 64 bits
def _mimage(d, L):
    return d - L * torch.round(d / L) if L else d


_ZERO = -(1 << 28)  # the exponent of a zero


class _Exchange:
    """V_B and forces of one system: the recursions over y_v = exp(-beta (V^{[1,v]} - C[v]))
    and their mirror image, every number as mantissa and exponent."""

    def __init__(self, pos, m, wP, beta, L=0.0):
        N, P, _ = pos.shape
        k = m * wP * wP
        r1, rP = pos[:, 0], pos[:, -1]
        d = _mimage(pos[:, 1:] - pos[:, :-1], L)
        self.Eint = 0.5 * k * d.square().sum((1, 2))
        F = torch.zeros_like(pos)
        F[:, :-1] += k * d
        F[:, 1:] -= k * d
        link = torch.zeros(N, dtype=torch.float64, device=pos.device)
        dl = _mimage(rP[:-1] - r1[1:], L)
        link[:-1] = 0.5 * k * dl.square().sum(1)
        inv_ln2 = 1.0 / math.log(2.0)
        x = beta * link * inv_ln2
        n = torch.floor(x)
        cm, ce = (torch.exp2(x - n).cpu().numpy() / np.arange(1, N + 1)).tolist(), n.long().tolist()
        C = (self.Eint + (x - n) * math.log(2.0) / beta).sum()
        B = max(1, min(N, (1 << 24) // N))  # rows of pair factors held at a time

        def factors(lo, hi, by_row):
            """g(a, b) for the rows b (or the columns a) lo..hi-1 against every partner; 0 unless a <= b."""
            own, oth = (rP, r1) if by_row else (r1, rP)
            d2 = _mimage(own[lo:hi, None] - oth[None], L).square().sum(2)
            x = (-beta * 0.5 * k * inv_ln2 * d2).clamp(min=float(_ZERO))
            e = torch.floor(x)
            i, j = torch.arange(lo, hi, device=pos.device)[:, None], torch.arange(N, device=pos.device)[None]
            mask = (j <= i) if by_row else (j >= i)
            return torch.exp2(x - e) * mask, e.int(), d2 * mask

        def row_sum(m, e, gm, ge):
            """sum of m 2^e g as (mantissa, exponent)."""
            e = e + ge
            top = int(e.max())
            f, x = math.frexp(float(np.ldexp(m * gm, np.maximum(e - top, -2000)).sum()))
            return f, top + x

        ym, ye = np.zeros(N + 1), np.full(N + 1, _ZERO, dtype=np.int32)
        ym[0], ye[0] = 0.5, 1
        for lo in range(0, N, B):
            gm, ge = (t.cpu().numpy() for t in factors(lo, min(N, lo + B), True)[:2])
            for v in range(lo, min(N, lo + B)):
                f, e = row_sum(ym[: v + 1], ye[: v + 1], gm[v - lo, : v + 1], ge[v - lo, : v + 1])
                f, up = math.frexp(f * cm[v])
                ym[v + 1], ye[v + 1] = f, e + ce[v] + up
        mm, me = np.zeros(N), np.full(N, _ZERO, dtype=np.int32)
        Bm, Be = np.zeros(N), np.full(N, _ZERO, dtype=np.int32)
        mm[N - 1], me[N - 1] = 0.5, 1
        for hi in range(N, 0, -B):
            lo = max(0, hi - B)
            gm, ge = (t.cpu().numpy() for t in factors(lo, hi, False)[:2])
            for a in range(hi - 1, lo - 1, -1):
                Bm[a], Be[a] = f, e = row_sum(mm[a:], me[a:], gm[a - lo, a:], ge[a - lo, a:])
                if a:
                    f, up = math.frexp(f * cm[a - 1])
                    mm[a - 1], me[a - 1] = f, e + ce[a - 1] + up
        ym, ye, mm, me, Bm, Be = (torch.from_numpy(t).to(pos.device) for t in (ym, ye, mm, me, Bm, Be))
        self.V = C - (torch.log(ym[N]) + (ye[N] - n.sum()) * math.log(2.0)) / beta
        # probabilities Pr[b -> a <= b], the direct links Pr[b -> b+1], and the exterior forces
        zm, ze = 1.0 / (ym[N] * N), -ye[N]
        direct = torch.zeros(N, dtype=torch.float64, device=pos.device)
        direct[:-1] = 1.0 - ym[1:N] * Bm[1:] * zm * torch.exp2((ye[1:N] + Be[1:] + ze).clamp(-2000, 900).to(torch.float64))
        spring = (direct * link).sum() + self.Eint.sum()
        rows, cols = torch.zeros_like(r1), torch.zeros_like(r1)
        for lo in range(0, N, B):
            hi = min(N, lo + B)
            gm, ge, d2 = factors(lo, hi, True)
            e = (ye[None, :N] + ge + me[lo:hi, None] + ze).clamp(-2000, 900)
            pr = ym[None, :N] * gm * mm[lo:hi, None] * zm * torch.exp2(e.to(torch.float64))
            d = _mimage(rP[lo:hi, None] - r1[None], L) * pr[:, :, None]
            rows[lo:hi] = d.sum(1)
            cols += d.sum(0)
            spring = spring + 0.5 * k * (pr * d2).sum()
        rows[:-1] += direct[:-1, None] * dl
        cols[1:] += direct[:-1, None] * dl
        F[:, -1] -= k * rows
        F[:, 0] += k * cols
        self.F, self.spring = F, spring


def _physical(pos, omega0, gauss, lj, L):
    """(U-bar, -grad U-bar): trap and pairs between beads of equal index, over P."""
    N, P, _ = pos.shape
    kt = omega0 * omega0
    U, F = 0.5 * kt * pos.square().sum(), -kt * pos
    if gauss or lj:
        per = max(1, min(P, (1 << 25) // (N * N)))
        for j in range(0, P, per):
            r = pos[:, j:j + per].transpose(0, 1)  # [beads][N][3]
            d = _mimage(r[:, :, None] - r[:, None], L)
            d2 = d.square().sum(3)
            off = 1.0 - torch.eye(N, dtype=torch.float64, device=pos.device)
            if gauss:
                e = gauss * torch.exp(-d2 / (2.0 * 0.25)) * off
                U = U + 0.5 * e.sum()
                f = ((e / 0.25)[..., None] * d).sum(2)
            else:
                eps, sig, rc = lj
                near = (d2 < rc * rc) & (off > 0)
                s6 = torch.where(near, sig * sig / torch.where(near, d2, 1.0), 0.0) ** 3
                c6 = (sig / rc) ** 6
                U = U + 0.5 * (4.0 * eps * ((s6 * s6 - s6) - near * (c6 * c6 - c6))).sum()
                f = ((24.0 * eps * (2.0 * s6 * s6 - s6) / torch.where(near, d2, 1.0))[..., None] * d).sum(2)
            F[:, j:j + per] += f.transpose(0, 1)
    return U / P, F / P


def _normals(count, step, seed):
    """Thermostat normals of elements 0..count-1: Philox4x32-10 words of the
    counter (element / 4, step), key seed, by Box-Muller."""
    mask = 0xFFFFFFFF
    blocks = (count + 3) // 4
    c = [torch.arange(blocks, dtype=torch.int64, device="cuda"), torch.full((blocks,), step & mask, device="cuda"),
         torch.full((blocks,), step >> 32, device="cuda"), torch.zeros(blocks, dtype=torch.int64, device="cuda")]
    k0, k1 = seed & mask, seed >> 32

    def mul(k, x):  # 32 x 32 -> (high, low) words
        lo, hi = k * (x & 0xFFFF), k * (x >> 16)
        t = hi + (lo >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    u = [(w.to(torch.float64) + 0.5) / 4294967296.0 for w in c]
    ra, rb = torch.sqrt(-2.0 * torch.log(u[0])), torch.sqrt(-2.0 * torch.log(u[2]))
    ta, tb = 2.0 * math.pi * u[1], 2.0 * math.pi * u[3]
    z = torch.stack([ra * torch.cos(ta), ra * torch.sin(ta), rb * torch.cos(tb), rb * torch.sin(tb)], 1)
    return z.reshape(-1)[:count]


def exact(case, seed):
    pos = _positions(case, seed)
    one = case["system"] != "replicas"
    if one:
        systems = [_sizes(case)]
        xs = [pos]
    else:
        systems = [(n, p, 1.0, math.sqrt(p) / b, b) for n, p, b in zip(*_replicas(case))]
        xs = list(pos)
    L = _box(case)
    if case["kind"] in ("forces", "autograd", "batch_forces"):
        got = [_Exchange(x, s[2], s[3], s[4], L) for x, s in zip(xs, systems)]
        if one:
            return {"V": got[0].V, "F" if case["kind"] == "forces" else "grad":
                    got[0].F if case["kind"] == "forces" else -got[0].F}
        return {"V": torch.stack([g.V for g in got]), "F": torch.cat([g.F.reshape(-1) for g in got])}
    vs = _velocities(case, seed, pos)
    vs = [vs] if one else vs
    helium, dt = case["system"] == "helium", case["dt"]
    count = sum(x.numel() for x in xs)

    def force(x, s):
        ex = _Exchange(x, s[2], s[3], s[4], L)
        U, F = _physical(x, 0.0 if helium else 1.0, case["gauss"], HE_LJ if helium else None, L)
        return ex, U, ex.F + F

    state = [force(x, s) for x, s in zip(xs, systems)]
    for step in range(case["steps"]):
        z, at = _normals(count, step, _seed_md(seed)), 0
        for i, s in enumerate(systems):
            x, v, F, m, beta = xs[i], vs[i], state[i][2], s[2], s[4]
            n, c1 = x.numel(), math.exp(-dt)
            c2 = math.sqrt((1.0 - c1 * c1) / (m * beta))
            v = v + 0.5 * dt / m * F
            x = x + 0.5 * dt * v
            v = c1 * v + c2 * z[at:at + n].reshape(x.shape)
            x = x + 0.5 * dt * v
            at += n
            state[i] = force(x, s)
            xs[i], vs[i] = x, v + 0.5 * dt / m * state[i][2]
    energies = []
    for x, v, s, (ex, U, _) in zip(xs, vs, systems, state):
        kin = 0.5 * s[2] * v.square().sum()
        energies.append(torch.stack([ex.V, U, kin, 1.5 * s[0] * s[1] / s[4] - ex.spring + U]))
    if one:
        return {"x": xs[0], "v": vs[0], "energies": energies[0]}
    return {"x": torch.cat([x.reshape(-1) for x in xs]), "v": torch.cat([v.reshape(-1) for v in vs]),
            "energies": torch.stack(energies)}
