"""The work that users of the TREE library have it do, as cases that can be timed.

Every case goes through the package's public entry points (``Context`` and the
``autograd`` front end), with state and results in CUDA tensors:

* ``force``    -- new positions in, accelerations and potentials out,
* ``block``    -- new state in, one or more blocks of the split-step push, the
                  energies and the advanced state out,
* ``vjp``      -- accelerations as a differentiable function of the positions and
                  the vector-Jacobian product of its backward pass,
* ``gradient`` -- electron kinetic energy after a run and its gradient with respect
                  to the initial state.

Contexts of either walk precision are used: FP64 contexts compute in 64 bits and
their results are kept as they are; FP32C contexts compute their forces in single
precision (the library's FP32 mode), so what the program keeps of them are
single-precision fields, gradients and snapshots.

``exact`` restates the method in plain float64 torch: octree from Morton cells,
moments straight from each box's particles, the per-particle opening criterion,
box by box and pair by pair, level by level.  It shares no code with the package.
"""
import math

import numpy as np
import torch

from paper_0709_3331_gb300 import UCP_FP32C, UCP_FP64, Context
from paper_0709_3331_gb300.autograd import electron_ke_after_run, tree_accel
from paper_0709_3331_gb300.inputs import batched_sizes

Q = (1.0, -1.0)          # ion, electron charge
M = (1000.0, 1.0)        # ion, electron mass
T_E, T_I = 1.0, 0.01     # temperatures of the initial velocities
EPS = 0.01
DT, K = 1e-3, 10         # electron step, electron steps per ion step
LAMBDA = 0.05            # Kelbg length of the cases that use that pair law


def listed():
    return [
        # the small standard workload: one force evaluation of 2,048 particles, where
        # latency and launches count (interactive use, parameter scans)
        dict(name="force_fp64_2k", kind="force", n=2048, sigma=1.0, theta=0.5, leaf_cap=8, fp64=True),
        # the same workload stepped: 10 velocity Verlet steps, ions every 10
        dict(name="block_fp64_2k", kind="block", n=2048, sigma=1.0, theta=0.5, leaf_cap=8, fp64=True,
             graphs=False),
        # the plain method at its standard size: one block of 10 electron steps in FP64
        dict(name="block_fp64_128k", kind="block", n=131072, sigma=4.0, theta=0.5, leaf_cap=32,
             fp64=True, graphs=False),
        # the accelerations inside a differentiable program, in FP64 (fits, gradient checks)
        dict(name="vjp_fp64_4k", kind="vjp", n=4096, sigma=1.3, theta=0.5, leaf_cap=16, fp64=True),
        # a small odd-sized cloud in the FP32 mode
        dict(name="force_fp32c_4k_odd", kind="force", n=4099, sigma=1.3, theta=0.5, leaf_cap=16,
             fp64=False),
        # high accuracy (theta 0.3) on an odd-sized cloud of ordinary size
        dict(name="force_fp32c_200k_t03", kind="force", n=200001, sigma=5.8, theta=0.3, leaf_cap=32,
             fp64=False),
        # one force evaluation of the headline workload
        dict(name="force_fp32c_512k", kind="force", n=524288, sigma=8.0, theta=0.5, leaf_cap=32,
             fp64=False),
        # the headline workload stepped: one block of 10 electron steps as a captured graph
        dict(name="block_fp32c_512k", kind="block", n=524288, sigma=8.0, theta=0.5, leaf_cap=32,
             fp64=False, graphs=True),
        # the largest cloud: production sizes beyond the standard workloads
        dict(name="force_fp32c_4m", kind="force", n=4194304, sigma=16.0, theta=0.5, leaf_cap=32,
             fp64=False),
        # the paper's own pair law (electron-ion Kelbg) at the paper's 1e5 particles
        dict(name="kelbg_fp32c_100k", kind="force", n=100000, sigma=4.6, theta=0.4, leaf_cap=32,
             fp64=False, kelbg=True),
        # the ensemble workload: 64 independent clouds of 4,096 to 65,536 particles,
        # one block of 10 electron steps for all of them
        dict(name="block_fp32c_64_clouds", kind="block", clouds=64, sizes_seed=4, theta=0.5,
             leaf_cap=32, fp64=False, graphs=True),
        # the differentiation workload: gradient through 20 electron steps, checkpoints
        # every 10, of 262,144 particles
        dict(name="gradient_fp32c_256k", kind="gradient", n=262144, sigma=6.0, theta=0.5, leaf_cap=32,
             fp64=False, steps=20, checkpoint=10),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["force"] * 4 + ["block"] * 3 + ["clouds", "vjp", "gradient"])
    fp64 = rng.random() < 0.35
    c = dict(kind=kind, theta=round(rng.uniform(0.3, 0.7), 3), leaf_cap=rng.choice([8, 16, 32]),
             fp64=fp64)
    if kind == "force":
        n = size(1000, 100000 if fp64 else 2000000)
        c["kelbg"] = rng.random() < 0.2
    elif kind == "block":
        n = size(1000, 30000 if fp64 else 500000)
        c["graphs"] = rng.random() < 0.5
    elif kind == "clouds":
        return dict(kind="block", clouds=rng.randint(3, 24), sizes_seed=rng.randint(5, 10**6), graphs=True,
                    theta=round(rng.uniform(0.45, 0.7), 3), leaf_cap=c["leaf_cap"], fp64=False)
    elif kind == "vjp":
        n = size(1000, 8000 if fp64 else 300000)
    else:
        n = size(2000, 150000)
        c.update(fp64=False, steps=10 * rng.randint(1, 3), checkpoint=10,
                 theta=round(rng.uniform(0.45, 0.7), 3))
    c["n"] = n
    c["sigma"] = round(8.0 * (n / 524288.0) ** (1.0 / 3.0), 3)
    return c


# ------------------------------------------------------------------ inputs
def _sizes(case):
    if "clouds" in case:
        return batched_sizes(case["clouds"], case["sizes_seed"])
    return [case["n"]], [case["sigma"]]


def _inputs(case, seed):
    """Gaussian clouds, half ions (first) and half electrons, Maxwellian velocities with
    each species' mean removed; clouds one after another."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    pos, vel, sp = [], [], []
    for n, sigma in zip(*_sizes(case)):
        ni = n // 2
        pos.append(torch.randn(n, 3, generator=g, dtype=torch.float64, device="cuda") * sigma)
        v = torch.randn(n, 3, generator=g, dtype=torch.float64, device="cuda")
        v[:ni] *= math.sqrt(T_I / M[0])
        v[ni:] *= math.sqrt(T_E / M[1])
        v[:ni] -= v[:ni].mean(0)
        v[ni:] -= v[ni:].mean(0)
        vel.append(v)
        s = torch.ones(n, dtype=torch.int8, device="cuda")
        s[:ni] = 0
        sp.append(s)
    pos, vel, sp = torch.cat(pos), torch.cat(vel), torch.cat(sp)
    lam = torch.randn(pos.shape, generator=g, dtype=torch.float64, device="cuda")
    return pos, vel, sp, lam


def prepare(case, seed):
    sizes, _ = _sizes(case)
    pos, vel, sp, lam = _inputs(case, seed)
    ctx = Context(pos.shape[0], Q, M, leaf_cap=case["leaf_cap"],
                  precision=UCP_FP64 if case["fp64"] else UCP_FP32C,
                  kelbg_lambda=LAMBDA if case.get("kelbg") else None,
                  sizes=sizes if "clouds" in case else None)
    if case.get("graphs"):
        ctx.set_graphs(True)
    st = dict(case=case, ctx=ctx, pos=pos, vel=vel, sp=sp)
    if case["kind"] == "force":
        st.update(acc=torch.empty_like(pos), phi=torch.empty_like(pos[:, 0]))
    elif case["kind"] == "block":
        st.update(pos1=torch.empty_like(pos), vel1=torch.empty_like(vel))
    elif case["kind"] == "vjp":
        st.update(lam=lam)
        pos.requires_grad_(True)
    else:
        pos.requires_grad_(True)
        vel.requires_grad_(True)
    return st


# ------------------------------------------------------------------ the pass
def run(st):
    case, ctx, pos, vel, sp = st["case"], st["ctx"], st["pos"], st["vel"], st["sp"]
    theta = case["theta"]
    keep = (lambda a: a) if case["fp64"] else _single
    if case["kind"] == "force":
        ctx.set_state(pos, vel, sp)
        ctx.tree_force(theta, EPS, st["acc"], st["phi"])
        return {"acc": keep(st["acc"]), "phi": keep(st["phi"])}
    if case["kind"] == "block":
        ctx.set_state(pos, vel, sp)
        ctx.step(DT, K, K, theta, EPS)
        e = ctx.energy_clouds(theta, EPS) if "clouds" in case else ctx.energy(theta, EPS)
        ctx.get_state(st["pos1"], st["vel1"])
        return {"pos": keep(st["pos1"]), "vel": keep(st["vel1"]), "energy": keep(e)}
    if case["kind"] == "vjp":
        acc = tree_accel(pos, sp, ctx, theta, EPS)
        mu, = torch.autograd.grad(acc, pos, st["lam"])
        return {"acc": keep(acc.detach()), "mu": keep(mu)}
    loss = electron_ke_after_run(pos, vel, sp, ctx, DT, K, case["steps"], theta, EPS, case["checkpoint"])
    gx, gv = torch.autograd.grad(loss, (pos, vel))
    return {"loss": keep(loss.detach()), "gx": keep(gx), "gv": keep(gv)}


def _single(a):
    return a.astype(np.float32) if isinstance(a, np.ndarray) else a.float()


# ------------------------------------------------------------------ the work
def work(case):
    """Interactions by a fit to the counts of the standard workloads (per target about 1250
    boxes and 780 pairs at theta 0.5 with 524,288 particles and leaves of 32); 64 and 20 flop
    each, three times that for their derivative.  Bytes: state in, results out."""
    sizes, _ = _sizes(case)
    f = 0.0
    for n in sizes:
        t = case["theta"]
        boxes = min(n / 2.0, 1250.0 * (0.5 / t) ** 2.1 * max(0.2, math.log(n / 500.0) / 6.95)
                    * (32.0 / case["leaf_cap"]) ** 0.1)
        pairs = min(float(n), 780.0 * (0.5 / t) ** 2.7 * (case["leaf_cap"] / 32.0) ** 0.85)
        one = n * (64.0 * boxes + 20.0 * pairs)
        walks = 1.0
        if case["kind"] == "block":
            walks = 2.0 + (K - 1) * 0.5          # first, last, and the electrons in between
        elif case["kind"] == "vjp":
            walks = 1.0 + 3.0
        elif case["kind"] == "gradient":
            s = case["steps"]
            fwd = s / K * (1.0 + (K - 1) * 0.5)
            walks = 2.0 * fwd + 3.0 * fwd        # the run, its recomputation, its adjoint
        f += walks * one
    n = float(sum(sizes))
    moved = {"force": 24 + 24 + 1 + 32, "block": 49 + 48, "vjp": 25 + 24 + 48, "gradient": 49 + 48}
    return {"bytes": n * moved[case["kind"]], "flops": f}


# ------------------------------------------------------------------ 64-bit restatement
class _Tree:
    """Octree of one cloud, as levels of boxes; moments differentiable in the positions."""

    def __init__(self, x, sp, leaf_cap):
        dev = x.device
        xd = x.detach()
        n = x.shape[0]
        mn, mx = xd.min(0).values, xd.max(0).values
        c = (mn + mx) * 0.5
        ext = float((mx - mn).max())
        L = ext * (1.0 + 2.0 ** -20) if ext > 0 else 1.0
        lo = c - L * 0.5
        k = ((xd - lo) * (2097152.0 / L)).to(torch.int64).clamp(0, 2097151)
        key = torch.zeros(n, dtype=torch.int64, device=dev)
        for b in range(21):
            for a in range(3):
                key |= ((k[:, a] >> b) & 1) << (3 * b + a)
        key, order = torch.sort(key, stable=True)
        self.order, self.x, self.n = order, x[order], n
        self.sp = sp[order].long()
        q = torch.tensor(Q, dtype=torch.float64, device=dev)[self.sp]
        self.q, aq = q, q.abs()
        self.levels = []
        inside = torch.arange(n, device=dev)           # particles whose box at this depth exists
        parent = torch.zeros(n, dtype=torch.int64, device=dev)
        for d in range(22):
            pre = key[inside] >> (3 * (21 - d)) if d else torch.zeros_like(inside)
            uniq, box, cnt = torch.unique_consecutive(pre, return_inverse=True, return_counts=True)
            nb = uniq.shape[0]
            start = torch.zeros(nb, dtype=torch.int64, device=dev)
            first = torch.cumsum(cnt, 0) - cnt
            start[:] = inside[first]
            s = L * 2.0 ** -d
            ic = torch.zeros(nb, 3, dtype=torch.int64, device=dev)
            for b in range(21):
                for a in range(3):
                    ic[:, a] |= ((uniq >> (3 * b + a)) & 1) << b
            z = lo + (ic.double() + 0.5) * s
            xs, qs, aqs = self.x[inside], q[inside], aq[inside]

            def add(v):
                return torch.zeros((nb,) + v.shape[1:], dtype=torch.float64, device=dev).index_add(0, box, v)

            S0, Mn = add(aqs), add(qs)
            e = add(aqs[:, None] * (xs - z[box])) / torch.where(S0 > 0, S0, torch.ones_like(S0))[:, None]
            cen = z + e
            y = xs - cen[box]
            qy = qs[:, None] * y
            D = add(qy)
            Qm = add(qy[:, :, None] * y[:, None, :])
            cd = cen.detach()
            w = cd - z
            delta = torch.sqrt((w[:, 0] * w[:, 0] + w[:, 1] * w[:, 1]) + w[:, 2] * w[:, 2])
            leaf = (cnt <= leaf_cap) | torch.full_like(cnt, d == 21, dtype=torch.bool)
            self.levels.append(dict(s=s, start=start, cnt=cnt, cen=cen, M=Mn, D=D, Q=Qm, delta=delta, leaf=leaf))
            if d:
                up = self.levels[d - 1]
                pb = parent[inside[first]]               # box of the level above
                kids = torch.bincount(pb, minlength=up["cnt"].shape[0])
                up["kids"], up["kid0"] = kids, torch.cumsum(kids, 0) - kids
            if bool(leaf.all()):
                break
            parent[inside] = box
            inside = inside[~leaf[box]]

    def field(self, theta, eps, lo, hi, kelbg=False):
        """E and phi at the particles lo .. hi of the sorted order."""
        dev = self.x.device
        xt = self.x[lo:hi]
        m = hi - lo
        E = torch.zeros(m, 3, dtype=torch.float64, device=dev)
        phi = torch.zeros(m, dtype=torch.float64, device=dev)
        t = torch.arange(m, device=dev)
        b = torch.zeros(m, dtype=torch.int64, device=dev)
        e2 = eps * eps
        for lv in self.levels:
            with torch.no_grad():
                r = xt[t] - lv["cen"][b]
                d2 = (r[:, 0] * r[:, 0] + r[:, 1] * r[:, 1]) + r[:, 2] * r[:, 2]
                if theta > 0:
                    rc = lv["s"] / theta + lv["delta"][b]
                    acc = rc * rc < d2
                else:
                    acc = torch.zeros_like(d2, dtype=torch.bool)
                del r, d2
            ta, ba = t[acc], b[acc]
            if ta.numel():
                r = xt[ta] - lv["cen"][ba]
                g = 1.0 / torch.sqrt((r * r).sum(1) + e2)
                u = g * g
                D, Qm = lv["D"][ba], lv["Q"][ba]
                QR = (Qm * r[:, None, :]).sum(2)
                tr = Qm[:, 0, 0] + Qm[:, 1, 1] + Qm[:, 2, 2]
                w = (D * r).sum(1) - 0.5 * tr
                h = u * (r * QR).sum(1)
                Mn = lv["M"][ba]
                phi = phi.index_add(0, ta, g * (Mn + u * (w + 1.5 * h)))
                g3 = g * u
                f = (g3 * (Mn + 3.0 * u * (w + 2.5 * h)))[:, None] * r - g3[:, None] * (D + 3.0 * u[:, None] * QR)
                E = E.index_add(0, ta, f)
                del r, g, u, D, Qm, QR, w, h, f
            lf = lv["leaf"][b]
            tl, bl = t[~acc & lf], b[~acc & lf]
            if tl.numel():
                cnt = lv["cnt"][bl]
                tp = torch.repeat_interleave(tl, cnt)
                off = torch.arange(tp.shape[0], device=dev) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
                j = torch.repeat_interleave(lv["start"][bl], cnt) + off
                other = j != tp + lo
                tp, j = tp[other], j[other]
                r = xt[tp] - self.x[j]
                rr = (r * r).sum(1)
                g = 1.0 / torch.sqrt(rr + e2)
                p, f = g, g * g * g
                if kelbg:
                    d = torch.sqrt(rr)
                    ex, ome = torch.exp(-d / LAMBDA), -torch.expm1(-d / LAMBDA)
                    unlike = self.sp[j] != self.sp[tp + lo]
                    f = torch.where(unlike, ome / (rr * d) - ex / (LAMBDA * rr), f)
                    p = torch.where(unlike, ome / d, p)
                phi = phi.index_add(0, tp, self.q[j] * p)
                E = E.index_add(0, tp, (self.q[j] * f)[:, None] * r)
                del r, rr, g, p, f
            if "kids" not in lv:
                break
            go = ~acc & ~lf
            t, b = t[go], b[go]
            if not t.numel():
                break
            kids = lv["kids"][b]
            t2 = torch.repeat_interleave(t, kids)
            off = torch.arange(t2.shape[0], device=dev) - torch.repeat_interleave(torch.cumsum(kids, 0) - kids, kids)
            b = torch.repeat_interleave(lv["kid0"][b], kids) + off
            t = t2
        return E, phi


def _accel(pos, sp, case, n, off=0):
    """a and phi in caller order of the cloud pos[off : off + n]."""
    x, s = pos[off:off + n], sp[off:off + n]
    T = _Tree(x, s, case["leaf_cap"])
    per = max(1024, int(16384 * (case["theta"] / 0.5) ** 2.5))
    parts = [T.field(case["theta"], EPS, lo, min(n, lo + per), case.get("kelbg", False)) for lo in range(0, n, per)]
    E, phi = torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])
    qm = T.q / torch.tensor(M, dtype=torch.float64, device=x.device)[T.sp]
    back = torch.empty_like(T.order)
    back[T.order] = torch.arange(n, device=x.device)
    return (qm[:, None] * E)[back], phi[back]


def exact(case, seed):
    pos, vel, sp, lam = _inputs(case, seed)
    if case["kind"] == "force":
        acc, phi = _accel(pos, sp, case, case["n"])
        return {"acc": acc, "phi": phi}
    if case["kind"] == "vjp" and case["n"] <= 20000:
        pos.requires_grad_(True)
        acc, _ = _accel(pos, sp, case, case["n"])
        mu, = torch.autograd.grad(acc, pos, lam)
        return {"acc": acc.detach(), "mu": mu}
    if case["kind"] == "block" and "clouds" not in case and case["n"] <= 40000:
        n = case["n"]
        ion, el = (sp == 0)[:, None].double(), (sp == 1)[:, None].double()
        a, _ = _accel(pos, sp, case, n)
        vel = vel + ion * (0.5 * K * DT) * a
        for _ in range(K):
            vel = vel + el * (0.5 * DT) * a
            pos = pos + DT * vel
            a, phi = _accel(pos, sp, case, n)
            vel = vel + el * (0.5 * DT) * a
        vel = vel + ion * (0.5 * K * DT) * a
        m = torch.tensor(M, dtype=torch.float64, device="cuda")[sp.long()]
        q = torch.tensor(Q, dtype=torch.float64, device="cuda")[sp.long()]
        ke = 0.5 * m * (vel * vel).sum(1)
        ki, kel, pe = float(ke[sp == 0].sum()), float(ke[sp == 1].sum()), float(0.5 * (q * phi).sum())
        P = float((m[:, None] * vel).sum(0).norm())
        return {"pos": pos, "vel": vel, "energy": np.array([ki, kel, pe, ki + kel + pe, P, float(K)])}
    return None  # gradients of runs, ensembles and long blocks: not in 20 seconds
