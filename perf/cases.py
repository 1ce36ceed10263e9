"""Performance cases: what a user of the hybrid tree library runs, through its public entry points.

One pass of a `step` case is one soft step (n_hard hard sub-steps, one tree build each) of a running simulation:
hybrid_step, or hybrid_step_batched for an ensemble; `calls` is one kick-drift-kick step driven from outside with the
single calls (drift, build, soft force, hard force, kicks); `energy` is the energy diagnostic; `serve` sends a mix of
requests through the server from host arrays to host arrays. States are returned in the particles' input order.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1406_6158_gb300 import hybrid

FIELDS = ("x", "y", "z", "vx", "vy", "vz", "m")
ACCS = ("ax_s", "ay_s", "az_s", "ax_h", "ay_h", "az_h")
DT = 1.0 / 512          # soft step of the workloads with a fixed step: a few % of the shortest orbital time
EXACT_MAX_N = 140000    # direct FP64 summation in torch stays within seconds up to here


# ---------------------------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest simulation anyone runs in earnest: every launch counts
        {"name": "step_4k", "kind": "step", "n": 4096, "model": "plummer", "split": "eps4", "eps": 1 / 64,
         "theta": 0.5, "n_hard": 4, "n_crit": 64, "tpg": 0, "depth": 0, "prec": 1},
        # the headline workload: one Plummer sphere of 2^17 particles with the autotuner's usual setting
        {"name": "step_131k", "kind": "step", "n": 1 << 17, "model": "plummer", "split": "eps4", "eps": 1 / 128,
         "theta": 0.5, "n_hard": 4, "n_crit": 128, "tpg": 32, "depth": 2, "prec": 1},
        # the largest single system: a cuspy halo, eight hard sub-steps, tighter opening angle
        {"name": "step_halo_16m", "kind": "step", "n": 1 << 24, "model": "hernquist", "split": "eps3",
         "eps": 1 / 512, "theta": 0.4, "n_hard": 8, "n_crit": 256, "tpg": 64, "depth": 2, "prec": 1},
        # an ensemble of uneven systems advanced together
        {"name": "step_batch_512", "kind": "batch", "count": 512, "lo": 10.0, "hi": 17.0, "sizes": 3, "theta": 0.5,
         "n_hard": 4, "n_crit": 256, "tpg": 64, "depth": 2},
        # the method's published parameters (absolute MAC, N-dependent softening and radii), a quarter of its step
        {"name": "step_absmac_1m", "kind": "step", "n": 1 << 20, "model": "plummer", "split": "paper", "n_hard": 4,
         "n_crit": 256, "tpg": 64, "depth": 2, "prec": 1},
        # the normal tree (no hard part): one build and one force per step, same parameters
        {"name": "step_normal_262k", "kind": "step", "n": 1 << 18, "model": "plummer", "split": "normal", "n_hard": 1,
         "n_crit": 128, "tpg": 32, "depth": 2, "prec": 1},
        # trees and neighbour lists reused across the hard sub-steps (Verlet skin)
        {"name": "step_skin_131k", "kind": "step", "n": 1 << 17, "model": "plummer", "split": "eps4", "eps": 1 / 128,
         "theta": 0.5, "n_hard": 4, "n_crit": 128, "tpg": 32, "depth": 2, "prec": 1, "skin": 0.00625},
        # an integrator of the user's own over the single calls, odd size, default stream (no captured graphs)
        {"name": "calls_100k", "kind": "calls", "n": 100003, "model": "plummer", "split": "eps4", "eps": 1 / 128,
         "theta": 0.5, "n_hard": 1, "n_crit": 64, "tpg": 0, "depth": 0, "prec": 1},
        # the plain method: FP64 throughout, small
        {"name": "step64_4k", "kind": "step", "n": 4096, "model": "plummer", "split": "eps4", "eps": 1 / 64,
         "theta": 0.5, "n_hard": 4, "n_crit": 64, "tpg": 0, "depth": 0, "prec": 0},
        # the plain method through the single calls, ragged size
        {"name": "calls64_30k", "kind": "calls", "n": 30011, "model": "plummer", "split": "eps4", "eps": 1 / 64,
         "theta": 0.5, "n_hard": 1, "n_crit": 64, "tpg": 0, "depth": 0, "prec": 0},
        # total energy by direct summation: the check a run makes every so often
        {"name": "energy_65k", "kind": "energy", "n": 1 << 16, "model": "plummer", "eps": 1 / 128},
        # continuous batching: requests of uneven size join, advance together and leave
        {"name": "serve_8", "kind": "serve", "count": 8, "lo": 12.0, "hi": 17.0, "sizes": 5, "theta": 0.5,
         "n_hard": 4, "n_crit": 128, "tpg": 32, "steps": 4},
    ]


def _log_n(rng, lo, hi):
    return int(2.0 ** rng.uniform(lo, hi)) | rng.randint(0, 1)


def draw(rng: random.Random):
    """One more case: single systems of 2^11 to 2^22.5 particles in every mode, ensembles, requests, energies."""
    kind = rng.choice(["step", "step", "step", "step", "batch", "calls", "energy", "serve"])
    if kind == "batch":
        lo = rng.uniform(10.0, 12.0)
        return {"kind": "batch", "count": rng.randint(16, 300), "lo": lo, "hi": rng.uniform(lo + 1.0, 16.5),
                "sizes": rng.randint(0, 1 << 20), "theta": rng.choice([0.4, 0.5, 0.6]), "n_hard": rng.choice([2, 4]),
                "n_crit": rng.choice([128, 256]), "tpg": rng.choice([32, 64]), "depth": rng.choice([0, 2, 4])}
    if kind == "energy":
        return {"kind": "energy", "n": _log_n(rng, 11.0, 16.5), "model": rng.choice(["plummer", "hernquist"]),
                "eps": 1 / 128}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(2, 9), "lo": 12.0, "hi": rng.uniform(14.0, 17.5),
                "sizes": rng.randint(0, 1 << 20), "theta": 0.5, "n_hard": rng.choice([2, 4]), "n_crit": 128,
                "tpg": 32, "steps": rng.randint(2, 6)}
    prec = 0 if rng.random() < 0.2 else 1
    c = {"kind": kind, "n": _log_n(rng, 11.0, 15.0 if prec == 0 else 18.0 if kind == "calls" else 22.5),
         "model": rng.choice(["plummer", "plummer", "hernquist"]), "prec": prec,
         "split": rng.choice(["eps4", "eps4", "eps3", "paper", "normal"]), "theta": rng.choice([0.4, 0.5, 0.6])}
    c["eps"] = 0.25 / c["n"] ** (1.0 / 3.0)
    c["n_hard"] = 1 if c["split"] == "normal" or kind == "calls" else rng.choice([2, 4, 8])
    c["n_crit"] = rng.choice([32, 64, 128, 256])
    c["tpg"] = rng.choice([0, c["n_crit"] // 4])
    c["depth"] = rng.choice([0, 2, 4])
    if kind == "step" and prec == 1 and c["split"] in ("eps4", "eps3") and c["n"] < 1 << 18 and rng.random() < 0.5:
        c["skin"] = 0.00625
    return c


# ---------------------------------------------------------------------------------------------------------------
# parameters and inputs
# ---------------------------------------------------------------------------------------------------------------
def _params(c, n=None):
    n = c["n"] if n is None else n
    kw = dict(n_hard=c["n_hard"], n_leaf=16, n_crit=c["n_crit"], threads_per_group=c["tpg"],
              tile_depth=c.get("depth", 0), precision=c.get("prec", 1), skin=c.get("skin", 0.0))
    split = c.get("split", "per_system")
    if split in ("paper", "normal"):    # eps = 0.1 N^-0.26, dt_h = eps / 2.6, R1 = 1.03 N^-1/3, a_err = 2^-8
        eps = 0.1 * n ** -0.26
        r1 = 0.0 if split == "normal" else 1.03 * n ** (-1.0 / 3.0)
        return hybrid.Params(eps=eps, R1=r1, R2=2.0 * r1, dt_soft=c["n_hard"] * eps / 2.6, mac=1, a_err=2.0 ** -8,
                             **kw)
    eps = 0.25 / n ** (1.0 / 3.0) if split == "per_system" else c["eps"]
    r1 = (3 if split == "eps3" else 4) * eps
    return hybrid.Params(eps=eps, theta=c["theta"], R1=r1, R2=2 * r1, dt_soft=DT, **kw)


def _sizes(c):
    r = random.Random(c["sizes"])
    return [int(2.0 ** r.uniform(c["lo"], c["hi"])) for _ in range(c["count"])]


def _directions(n, g, dev):
    cth = 2.0 * torch.rand(n, generator=g, device=dev, dtype=torch.float64) - 1.0
    phi = 2.0 * math.pi * torch.rand(n, generator=g, device=dev, dtype=torch.float64)
    sth = torch.sqrt(1.0 - cth * cth)
    return torch.stack([sth * torch.cos(phi), sth * torch.sin(phi), cth])


def _spheres(sizes, model, seed, dev="cuda"):
    """[7, sum(sizes)] FP64: spheres in equilibrium (G = M = a = 1, centre-of-mass frame) back to back.

    Plummer: radii from the enclosed mass (up to 0.999), speeds by rejection from q^2 (1 - q^2)^(7/2). Hernquist,
    truncated at 100: speeds from the isotropic Jeans dispersion, below the escape speed."""
    n = sum(sizes)
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    u = torch.rand(n, generator=g, device=dev, dtype=torch.float64)
    if model == "plummer":
        r = 1.0 / torch.sqrt((1.0 - u).clamp(1e-9, 0.999) ** (-2.0 / 3.0) - 1.0)
        q = torch.zeros(n, device=dev, dtype=torch.float64)
        todo = torch.arange(n, device=dev)
        while todo.numel():
            a = torch.rand(todo.numel(), generator=g, device=dev, dtype=torch.float64)
            b = 0.1 * torch.rand(todo.numel(), generator=g, device=dev, dtype=torch.float64)
            ok = b < a * a * (1.0 - a * a) ** 3.5
            q[todo[ok]] = a[ok]
            todo = todo[~ok]
        vel = q * math.sqrt(2.0) * (1.0 + r * r) ** -0.25 * _directions(n, g, dev)
    else:
        s = torch.sqrt(u) * (100.0 / 101.0)
        r = s / (1.0 - s)
        p = r + 1.0
        sig2 = (r * p ** 3 * torch.log1p(1.0 / r) - r / (12.0 * p) * (25.0 + r * (52.0 + r * (42.0 + r * 12.0))))
        vel = torch.sqrt(sig2.clamp(min=1e-6)) * torch.randn(3, n, generator=g, device=dev, dtype=torch.float64)
        speed = torch.linalg.vector_norm(vel, dim=0)
        vel = vel * torch.minimum(torch.ones_like(r), 0.95 * torch.sqrt(2.0 / p) / speed)
    out = torch.empty(7, n, device=dev, dtype=torch.float64)
    out[:3] = r * _directions(n, g, dev)
    out[3:6] = vel
    a = 0
    for k in sizes:
        out[:6, a:a + k] -= out[:6, a:a + k].mean(dim=1, keepdim=True)
        out[6, a:a + k] = 1.0 / k
        a += k
    return out


class _Batch:
    """Systems whose arrays are slices of one block: state [7, N], acc [6, N], id [N]."""

    def __init__(self, sizes, params, model, seed, own_stream):
        n = sum(sizes)
        prec = params[0].precision
        self.state = _spheres(sizes, model, seed)
        self.acc = torch.zeros(6, n, device="cuda", dtype=torch.float32 if prec else torch.float64)
        self.id = torch.cat([torch.arange(k, dtype=torch.int32) for k in sizes]).cuda()
        self.start = torch.cat([torch.full((k,), a, dtype=torch.int64) for k, a in
                                zip(sizes, np.cumsum([0] + sizes[:-1]).tolist())]).cuda()
        self.systems, a = [], 0
        host = np.zeros(max(sizes))
        for k, p in zip(sizes, params):
            s = hybrid.System({f: host[:k] for f in FIELDS}, precision=prec, params=p if len(sizes) > 1 else None)
            s.t.update({f: self.state[i, a:a + k] for i, f in enumerate(FIELDS)})
            s.t.update({f: self.acc[i, a:a + k] for i, f in enumerate(ACCS)})
            s.t["id"] = self.id[a:a + k]
            s.refresh()
            self.systems.append(s)
            a += k
        torch.cuda.synchronize()
        self.stream = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
        self.ctx = hybrid.Context(params[0], self.stream)
        self.dt = params[0].dt_soft

    def in_input_order(self):
        at = self.start + self.id
        state, acc = torch.empty_like(self.state), torch.empty_like(self.acc)
        state.index_copy_(1, at, self.state)
        acc.index_copy_(1, at, self.acc)
        return {"pos": state[:3], "vel": state[3:6], "mass": state[6], "acc_soft": acc[:3], "acc_hard": acc[3:]}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        sizes = _sizes(case)
        flat = _spheres(sizes, "plummer", seed).cpu().numpy()
        cut = np.cumsum([0] + sizes)
        states = [{f: np.ascontiguousarray(flat[i, a:b]) for i, f in enumerate(FIELDS)}
                  for a, b in zip(cut[:-1], cut[1:])]
        return {"kind": kind, "states": states, "steps": case["steps"], "params": [_params(case, k) for k in sizes],
                "server": hybrid.Server(_params(case, 1 << 16), 150e9, torch.cuda.Stream())}
    if kind == "energy":
        b = _Batch([case["n"]], [hybrid.Params(eps=case["eps"])], case["model"], seed, True)
        return {"kind": kind, "batch": b}
    sizes = _sizes(case) if kind == "batch" else [case["n"]]
    params = [_params(case, k) for k in sizes]
    b = _Batch(sizes, params, case.get("model", "plummer"), seed, kind != "calls")
    if kind == "calls":
        s = b.systems[0]
        b.ctx.hybrid_build_tree(s)
        b.ctx.hybrid_soft_force(s)
        b.ctx.hybrid_hard_force(s)
    else:
        b.ctx.hybrid_step_batched(b.systems, 0)     # the first forces of a run
    return {"kind": kind, "batch": b}


def run(state):
    kind = state["kind"]
    if kind == "serve":
        srv, out = state["server"], [None] * len(state["states"])
        todo = done = 0
        while done < len(out):
            for _ in range(2):                      # two requests arrive per server step
                if todo < len(out):
                    srv.submit(todo, state["states"][todo], state["params"][todo], state["steps"])
                    todo += 1
            srv.step()
            while (r := srv.next()) is not None:
                out[r[0]] = r[1]
                done += 1
        return out
    b = state["batch"]
    s = b.systems[0]
    if kind == "energy":
        return {"energy": np.array(b.ctx.hybrid_energy(s))}
    with torch.cuda.stream(b.stream):
        if kind == "calls":
            for which in (0, 1):
                b.ctx.hybrid_kick(s, which, 0.5 * b.dt)
            b.ctx.hybrid_drift(s, b.dt)
            b.ctx.hybrid_build_tree(s)
            b.ctx.hybrid_soft_force(s)
            b.ctx.hybrid_hard_force(s)
            for which in (0, 1):
                b.ctx.hybrid_kick(s, which, 0.5 * b.dt)
        elif kind == "batch":
            b.ctx.hybrid_step_batched(b.systems, 1)
        else:
            b.ctx.hybrid_step(s, 1)
        return b.in_input_order()


# ---------------------------------------------------------------------------------------------------------------
# what a pass cannot do without, and its values in 64 bits
# ---------------------------------------------------------------------------------------------------------------
def work(case):
    """State and accelerations read and written once; 20 floating-point operations per far pair and 26 per near pair
    (with the pair counts per particle that the opening angles give, 210 to 340 far pairs per halving of the system
    and about 400 near ones), 24 per pair of the direct energy sum."""
    kind = case["kind"]
    if kind == "energy":
        return {"bytes": 7 * 8 * case["n"], "flops": 12.0 * case["n"] ** 2}
    n = sum(_sizes(case)) if "count" in case else case["n"]
    each = n / case["count"] if "count" in case else n
    steps = case.get("steps", 1)
    acc = 48 if case.get("prec", 1) == 0 else 24
    far = 210.0 * (0.5 / case.get("theta", 0.5)) ** 2 * math.log2(each)
    near = 0.0 if case.get("split") == "normal" else 400.0
    nbytes = n * (2 * 56 if kind == "serve" else 2 * (56 + acc))
    return {"bytes": float(nbytes), "flops": steps * n * (20.0 * far + 26.0 * near * case["n_hard"])}


def _direct(pos, m, eps, r1, r2, soft):
    """Softened forces (G = 1) of the split by direct FP64 summation: (soft or None, hard), [3, n] each."""
    n = pos.shape[1]
    a_s, a_h = torch.zeros_like(pos), torch.zeros_like(pos)
    step = max(1, (1 << 26) // n)
    for i in range(0, n, step):
        d = [pos[k][None, :] - pos[k, i:i + step, None] for k in range(3)]
        r2s = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        if r2 > 0.0:
            y = ((r2 - torch.sqrt(r2s)) / (r2 - r1)).clamp_(0.0, 1.0)
            y2 = y * y
            w = y2 * y2 * y2 * (10.0 + y2 * (-15.0 + 6.0 * y2))
        else:
            w = torch.zeros_like(r2s)
        f = m[None, :] * torch.rsqrt(r2s + eps * eps) ** 3
        for k in range(3):
            fk = f * d[k]
            h = (fk * w).sum(dim=1)
            a_h[k, i:i + step] = h
            if soft:
                a_s[k, i:i + step] = (fk * (1.0 - w)).sum(dim=1)
    return (a_s if soft else None), a_h


def exact(case, seed):
    """Direct summation and the same leap-frog in FP64 (soft forces differ from the tree's by the tree's own error)."""
    kind = case["kind"]
    if kind == "energy":
        s = _spheres([case["n"]], case["model"], seed)
        pos, m, n = s[:3], s[6], case["n"]
        w = 0.0
        step = max(1, (1 << 26) // n)
        for i in range(0, n, step):
            d = pos[:, None, :] - pos[:, i:i + step, None]
            q = m[None, :] * torch.rsqrt((d * d).sum(dim=0) + case["eps"] ** 2)
            j = torch.arange(i, min(n, i + step), device=q.device)
            q[j - i, j] = 0.0
            w += float((q.sum(dim=1) * m[i:i + step]).sum())
        return {"energy": np.array([0.5 * float((m * (s[3:6] ** 2).sum(dim=0)).sum()), -0.5 * w])}
    if kind in ("batch", "serve") or case["n"] * math.sqrt(case["n_hard"]) > 2 * EXACT_MAX_N:
        return None
    p = _params(case)
    s = _spheres([case["n"]], case["model"], seed)
    pos, vel, m = s[:3].clone(), s[3:6].clone(), s[6]

    def forces(soft=True):
        return _direct(pos, m, p.eps, p.R1, p.R2, soft)

    a_s, a_h = forces()
    vel += 0.5 * p.dt_soft * a_s
    dt = p.dt_soft / p.n_hard
    for k in range(p.n_hard):
        vel += 0.5 * dt * a_h
        pos += dt * vel
        a_s, a_h = forces(k == p.n_hard - 1)
        vel += 0.5 * dt * a_h
    vel += 0.5 * p.dt_soft * a_s
    return {"pos": pos, "vel": vel, "mass": m, "acc_soft": a_s, "acc_hard": a_h}
