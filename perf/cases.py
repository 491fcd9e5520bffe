"""Workloads of the tree gravity and collision library, each through its public
Python entry points (``paper_1110_4876_gb300.rb``).

A case is one call pattern of a user's program: particles in host memory are
given to a simulation that the program keeps, some steps are taken (or the
forces evaluated, or the network trained), and the result is read back into
host memory.  Particle counts run from the 2400-particle sheet, where launches
and latency are the cost, to the 1,000,000-particle sheet of the benchmark.

``exact`` computes the same results in plain 64-bit torch: its own tree walk
(the octree's cells level by level), pair search and pair-by-pair resolution.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1110_4876_gb300 import inputs as I
from paper_1110_4876_gb300 import learned
from paper_1110_4876_gb300 import rb

STATE = ("x", "y", "z", "vx", "vy", "vz")
FIELDS = STATE + ("m", "r")
WALKS = {"fp32": rb.RB_WALK_FP32, "fp64": rb.RB_WALK_FP64, "learned": rb.RB_WALK_FP32_LEARNED}
TAU = 0.75            # optical depth N pi R^2 / (Lx Ly) of the benchmark's sheets
V_C, P_EPS = 7.7e-5, 0.234   # power-law restitution of the benchmark
THETA_FB = 0.5        # opening angle above which the network corrects a cell


def listed():
    return [
        # the small sheet (100 m, 2400 particles), four steps between outputs: launches and latency
        dict(name="sheet_2400", kind="sheet", n=2400, steps=4, theta=0.5, walk="fp32"),
        # a sheet with the options of a ring study: power-law restitution, half of the
        # particles massless tracers, a wider opening angle
        dict(name="sheet_20k_options", kind="sheet", n=19997, steps=2, theta=0.6, walk="fp32", law="power",
             tracers=True),
        # a monitored run: two steps, then the energy and momentum terms and the particles
        dict(name="sheet_30k_monitored", kind="sheet", n=30011, steps=2, theta=0.5, walk="fp32", energy=True),
        # the mid sheet (650 m, 100,000 particles)
        dict(name="sheet_100k", kind="sheet", n=100_000, steps=2, theta=0.5, walk="fp32"),
        # the benchmark's sheet, one step end to end through host buffers
        dict(name="sheet_1m", kind="sheet", n=1_000_000, steps=1, theta=0.5, walk="fp32"),
        # the FP64 walk, used to check a run's forces
        dict(name="sheet_65k_fp64", kind="sheet", n=65_537, steps=1, theta=0.5, walk="fp64"),
        # the learned far-field correction at its wide opening angle
        dict(name="sheet_20k_learned", kind="sheet", n=20_000, steps=2, theta=0.8, walk="learned"),
        # force evaluation of a star cluster for a caller's own integrator (open box, softened)
        dict(name="plummer_131k_forces", kind="plummer", n=1 << 17, theta=0.7, walk="fp32"),
        # elongated ring segment, plane sweep, no self-gravity
        dict(name="ring_300k_sweep", kind="ring", n=300_001, steps=2, detector="sweep"),
        # square sheet, collisions only, tree search
        dict(name="sheet_250k_collisions", kind="sheet", n=250_000, steps=2, theta=0.5, walk="fp32", gravity=False),
        # an ensemble of small boxes of differing size and density advanced together
        dict(name="ensemble_16", kind="ensemble", boxes=16, nmax=20000, steps=4, theta=0.5, walk="fp32"),
        # training of the correction network on residual samples
        dict(name="train_60k", kind="train", rows=60_000, epochs=2, batch=2048),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sheet", "sheet", "sheet", "sheet", "fp64", "learned", "plummer", "ring", "collisions", "box",
                       "ensemble", "train"])
    if kind == "sheet":
        n = _log(rng, 600, 1_000_000)
        c = dict(kind="sheet", n=n, steps=4 if n < 10_000 else 2 if n < 400_000 else 1, theta=rng.choice([0.4, 0.5, 0.6, 0.7]),
                 walk="fp32")
        if n > 600_000:
            c["theta"] = max(c["theta"], 0.5)
        if rng.random() < 0.25:
            c["law"] = "power"
        if rng.random() < 0.25:
            c["tracers"] = True
        if rng.random() < 0.2 and n < 30_000:
            c["energy"] = True
        return c
    if kind == "fp64":
        return dict(kind="sheet", n=_log(rng, 600, 70_000), steps=1, theta=rng.choice([0.5, 0.7]), walk="fp64")
    if kind == "learned":
        return dict(kind="sheet", n=_log(rng, 600, 60_000), steps=2, theta=0.8, walk="learned")
    if kind == "plummer":
        return dict(kind="plummer", n=_log(rng, 1000, 1 << 17), theta=rng.choice([0.5, 0.7, 0.9]), walk="fp32")
    if kind == "ring":
        return dict(kind="ring", n=_log(rng, 2000, 600_000), steps=2, detector=rng.choice(["sweep", "tree"]))
    if kind == "collisions":
        return dict(kind="sheet", n=_log(rng, 2000, 900_000), steps=2, theta=0.5, walk="fp32", gravity=False)
    if kind == "box":
        return dict(kind="box", n=_log(rng, 600, 40_000), steps=2, theta=0.6, walk="fp32",
                    quadrupole=rng.random() < 0.7)
    if kind == "ensemble":
        return dict(kind="ensemble", boxes=rng.randint(2, 16), nmax=_log(rng, 1500, 20000), steps=4, theta=0.5,
                    walk="fp32")
    return dict(kind="train", rows=_log(rng, 3000, 60_000), epochs=rng.randint(1, 2), batch=rng.choice([2048, 4096]))


# ---- inputs -----------------------------------------------------------------

def _weights(seed):
    """Network weights of the size training gives (He-normal layers, an output layer of a few per cent)."""
    g = np.random.default_rng([int(seed), 77])
    w = learned.init_weights(int(seed))
    w[-(64 * 3 + 3):-3] = g.normal(0.0, 0.004, 64 * 3)
    return w


def _boxes(case, seed):
    """[(box sides, Particles)] of a case."""
    seed = int(seed)
    n = case.get("n", 0)
    if case["kind"] == "sheet":
        L = math.sqrt(n * math.pi * I.RADIUS ** 2 / TAU)
        return [((L, L, L), I.sheet(L, n, seed))]
    if case["kind"] == "ring":
        Lx = I.long_sheet_size(n, tau=TAU)
        return [((Lx, 20.0, Lx), I.sheet_xy(Lx, 20.0, n, seed))]
    if case["kind"] == "plummer":
        return [((128.0,) * 3, I.plummer(n, seed))]
    if case["kind"] == "box":
        # granular gas in a periodic cube, volume fraction 0.05
        g = np.random.default_rng(seed)
        L = (n * 4.0 / 3.0 * math.pi / 0.05) ** (1.0 / 3.0)
        pos = g.uniform(-0.5 * L, 0.5 * L, (3, n))
        vel = g.normal(0.0, 1.0, (3, n))
        return [((L, L, L), I.Particles(*pos, *vel, np.full(n, 1.0), g.uniform(0.8, 1.0, n)))]
    return [((L, L, L), I.sheet(L, nb, 1000 * seed + k))
            for k, (nb, L, _) in enumerate(I.ensemble_boxes(case["boxes"], nmax=case["nmax"]))]


def _config(case, seed, box):
    kind = case["kind"]
    t0 = float(np.random.default_rng([int(seed), 5]).uniform(0.0, 5e4))
    if kind == "plummer":
        return dict(G=1.0, box=box, boundary=rb.RB_BC_OPEN, integrator=rb.RB_INT_LEAPFROG, theta=case["theta"],
                    softening=1e-3, dt=1e-3, gravity=1, collisions=0, walk=WALKS[case["walk"]])
    if kind == "box":
        return dict(G=1e-3, box=box, boundary=rb.RB_BC_PERIODIC, z_periodic=1, nghost=(1, 1, 1),
                    integrator=rb.RB_INT_LEAPFROG, theta=case["theta"], eps=0.8, dt=0.02, gravity=1,
                    quadrupole=int(case["quadrupole"]), collisions=rb.RB_COLL_TREE, walk=WALKS[case["walk"]])
    gravity = kind != "ring" and case.get("gravity", True)
    sweep = case.get("detector") == "sweep"
    return dict(G=I.G_SI, omega=I.OMEGA, box=box, nghost=(1, 1, 0), boundary=rb.RB_BC_SHEAR,
                integrator=rb.RB_INT_SEI, theta=case.get("theta", 0.5), eps=I.EPS_SHEET, dt=I.DT_SHEET, t0=t0,
                gravity=int(gravity), collisions=rb.RB_COLL_SWEEP if sweep else rb.RB_COLL_TREE,
                walk=WALKS[case.get("walk", "fp32")])


def _rows(case, seed):
    """Residual samples: the network's 12 inputs over their ranges and a smooth residual of a few per cent."""
    g = np.random.default_rng(int(seed))
    n = case["rows"]
    u = g.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    wr = g.uniform(0.5, 0.8, n)
    off = g.uniform(-0.3, 0.3, (n, 3))
    q = g.uniform(-0.1, 0.1, (n, 4))
    X = np.concatenate([u, wr[:, None], g.uniform(0.3, 5.0, (n, 1)), off, q], axis=1)
    Y = 0.05 * wr[:, None] ** 3 * (u * q[:, :1] + off * (u * off).sum(1, keepdims=True)) + g.normal(0, 1e-3, (n, 3))
    return X.astype(np.float32), Y.astype(np.float32)


def _pinned(n):
    return torch.empty(n, dtype=torch.float64, pin_memory=torch.cuda.is_available()).numpy()


def prepare(case, seed):
    if case["kind"] == "train":
        X, Y = _rows(case, seed)
        return dict(case=case, X=X, Y=Y, w=learned.init_weights(int(seed)), seed=int(seed) % 1000)
    boxes = _boxes(case, seed)
    sim = rb.Sim(nbox=len(boxes), **_config(case, seed, boxes[0][0]))
    whole = {k: _pinned(sum(P.n for _, P in boxes)) for k in FIELDS}
    src, out, at = [], [], 0
    for b, (L, P) in enumerate(boxes):
        if len(boxes) > 1:
            sim.set_box(b, L)
        # a program that exchanges particles with the library keeps them in pinned memory
        held = []
        for a in P.arrays():
            p = _pinned(P.n)
            p[:] = a
            held.append(p)
        src.append(held)
        out.append({k: whole[k][at: at + P.n] for k in FIELDS})
        at += P.n
        sim.set_particles(held, b)
    if case.get("walk") == "learned":
        rb.rb_load_mlp(sim.h, _weights(seed), THETA_FB)
    if case.get("law") == "power":
        rb.rb_set_restitution(sim.h, rb.RB_EPS_POWER, V_C, P_EPS)
    if case.get("tracers"):
        rb.rb_set_n_active(sim.h, case["n"] // 2)
    rb.rb_autotune(sim.h)
    return dict(case=case, sim=sim, src=src, out=out, whole=whole)


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        w, loss = rb.rb_mlp_train(state["X"], state["Y"], state["w"], epochs=case["epochs"], batch=case["batch"],
                                  lr=1e-3, seed=state["seed"])
        return dict(w=w, loss=loss)
    sim = state["sim"]
    for b, held in enumerate(state["src"]):
        sim.set_particles(held, b)
    if case["kind"] == "plummer":
        return dict(a=sim.gravity())
    sim.step(case["steps"])
    for b, out in enumerate(state["out"]):
        sim.particles(b, out)
    got = {k: state["whole"][k] for k in STATE}   # every box's particles, box after box
    if case.get("energy"):
        K, U, W, P = sim.energy_terms()
        got["terms"] = [K, U, W]
        got["momentum"] = P
    return got


# ---- what a pass cannot do without ------------------------------------------

def work(case):
    if case["kind"] == "train":
        # forward, backward by inputs and by weights: 2 flops each for 9347 weights
        n = case["rows"] * case["epochs"]
        return dict(bytes=15 * 4.0 * n, flops=6.0 * 9152 * n)
    if case["kind"] == "ensemble":
        n = case["boxes"] * (case["nmax"] - 500) / math.log(case["nmax"] / 500.0)
    else:
        n = case["n"]
    steps = case.get("steps", 1)
    bytes_ = n * (64.0 + (24.0 if case["kind"] == "plummer" else 48.0))
    flops = 200.0 * n * steps   # drift, kick, overlap tests, impulses
    if case["kind"] != "ring" and case.get("gravity", True):
        # accepted cells (60 flops), exact terms (20) and opening tests (10) of a Barnes-Hut
        # walk: about (8 / theta^2) log2 n opened shells with 9 images of a sheet
        th = case["theta"]
        terms = (2.0 / th ** 2 + 3.0) * (3.0 if case["kind"] in ("box", "plummer") else 1.0) * 4.0 * max(
            math.log2(n / max(1, case.get("boxes", 1))) - 6.0, 2.0)
        flops += n * steps * terms * (60.0 + 14.0)
        if case.get("walk") == "learned":
            flops += n * steps * 60.0 * 2.0 * 9152
    return dict(bytes=bytes_, flops=flops)


def tolerance(case):
    # about four times the differences seen between the launch shapes (other orders of the same sums);
    # the sheets' start holds deeply overlapping pairs, whose strong mutual pull magnifies rounding
    if case["kind"] == "train":
        return dict(rel=2e-4, max=4e-3)
    if case["kind"] == "plummer":
        return dict(rel=3e-7, max=8e-6)
    if case.get("walk") == "learned":
        return dict(rel=8e-5, max=1e-3)
    if case.get("walk") == "fp64" or case["kind"] == "ring" or not case.get("gravity", True):
        return dict(rel=1e-13, max=1e-11)
    return dict(rel=4e-6, max=4e-4)


# ---- the same in 64 bits ----------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _spread(v):
    x = v & 0x1FFFFF
    for s, m in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F), (4, 0x10C30C30C30C30C3),
                 (2, 0x1249249249249249)):
        x = (x | (x << s)) & m
    return x


class _Octree:
    """Cells of every depth with their mass, centre of mass and traceless quadrupole."""

    def __init__(self, pos, src, L):
        k = torch.floor((pos + 0.5 * L) / L * 2097152.0).clamp(0, 2097151).long()
        code = (_spread(k[:, 0]) << 2) | (_spread(k[:, 1]) << 1) | _spread(k[:, 2])
        code, self.order = torch.sort(code)
        self.pos, self.m = pos[self.order], src[self.order]
        self.L, self.levels = L, []
        inv_next = None
        for v in range(21, -1, -1):
            _, inv, cnt = torch.unique_consecutive(code >> (3 * (21 - v)), return_inverse=True, return_counts=True)
            first = torch.cumsum(cnt, 0) - cnt
            nc = len(cnt)
            lo = torch.floor((self.pos[first] + 0.5 * L) / L * 2.0 ** v) * (L / 2.0 ** v) - 0.5 * L
            M = torch.zeros(nc, dtype=pos.dtype, device=pos.device).index_add_(0, inv, self.m)
            rel = self.pos - lo[inv]
            S = torch.zeros(nc, 3, dtype=pos.dtype, device=pos.device).index_add_(0, inv, self.m[:, None] * rel)
            com = lo + torch.where(M[:, None] > 0, S / M[:, None].clamp_min(1e-300), torch.full_like(S, 0.5 * L / 2.0 ** v))
            d = self.pos - com[inv]
            d2 = (d * d).sum(1)
            q = torch.stack([3 * d[:, 0] ** 2 - d2, 3 * d[:, 1] ** 2 - d2, 3 * d[:, 2] ** 2 - d2, 3 * d[:, 0] * d[:, 1],
                             3 * d[:, 0] * d[:, 2], 3 * d[:, 1] * d[:, 2]], 1) * self.m[:, None]
            Q = torch.zeros(nc, 6, dtype=pos.dtype, device=pos.device).index_add_(0, inv, q)
            lev = dict(w=L / 2.0 ** v, cnt=cnt, first=first, lo=lo, M=M, com=com, Q=Q)
            if inv_next is not None:
                lev["child"] = inv_next[first]
                lev["nchild"] = inv_next[first + cnt - 1] - inv_next[first] + 1
            self.levels.insert(0, lev)
            inv_next = inv


def _expand(rows, begin, count):
    """Each row repeated count times, with begin, begin + 1, ... beside it."""
    at = torch.repeat_interleave(torch.arange(len(count), device=count.device), count)
    off = torch.arange(len(at), device=count.device) - (torch.cumsum(count, 0) - count)[at]
    return [r[at] for r in rows], begin[at] + off


def _network(w, X):
    w = torch.as_tensor(w, dtype=torch.float64, device=X.device)
    h, at = X, 0
    for a, b in ((12, 64), (64, 64), (64, 64), (64, 3)):
        W = w[at: at + a * b].reshape(a, b)
        h = h @ W + w[at + a * b: at + a * b + b]
        at += a * b + b
        if b == 64:
            h = torch.nn.functional.gelu(h, approximate="tanh")
    return h


def _forces(pos, src, box, offsets, G, theta, soft, quad, w_mlp=None, potential=False):
    """Barnes-Hut accelerations (and potentials) of every particle over the ghost images."""
    T = _Octree(pos, src, box[0])
    n = len(pos)
    acc = torch.zeros(n, 3, dtype=pos.dtype, device=pos.device)
    phi = torch.zeros(n, dtype=pos.dtype, device=pos.device)
    inside_rule = theta * theta > 1.0 / 3.0
    chunk = 1 << 17
    for o in offsets:
        tp_all = T.pos - torch.tensor(o, dtype=pos.dtype, device=pos.device)
        central = all(v == 0.0 for v in o) and o is offsets[len(offsets) // 2]
        for t0 in range(0, n, chunk):
            t = torch.arange(t0, min(n, t0 + chunk), device=pos.device)
            c = torch.zeros_like(t)
            for v, lev in enumerate(T.levels):
                if len(t) == 0:
                    break
                if v == 21:   # coincident at the depth limit: particle by particle
                    (t,), p = _expand([t], lev["first"][c], lev["cnt"][c])
                    one = torch.ones_like(t, dtype=torch.bool)
                else:
                    one = lev["cnt"][c] == 1
                    p = lev["first"][c]
                tt, pp = t[one], p[one]
                if central:
                    keep = tt != pp
                    tt, pp = tt[keep], pp[keep]
                d = T.pos[pp] - tp_all[tt]
                inv = 1.0 / torch.sqrt((d * d).sum(1) + soft * soft)
                acc.index_add_(0, tt, (T.m[pp] * inv ** 3)[:, None] * d)
                phi.index_add_(0, tt, -T.m[pp] * inv)
                if v == 21:
                    break
                t, c = t[~one], c[~one]
                d = lev["com"][c] - tp_all[t]
                r2 = (d * d).sum(1)
                ok = (lev["w"] ** 2 < theta * theta * r2) & (lev["nchild"][c] > 1)
                if inside_rule:
                    u = tp_all[t] - lev["lo"][c]
                    ok &= ~((u >= 0) & (u <= lev["w"])).all(1)
                ta, ca, da, ra = t[ok], c[ok], d[ok], r2[ok]
                M, Q = lev["M"][ca], lev["Q"][ca]
                inv = 1.0 / torch.sqrt(ra)
                invs = 1.0 / torch.sqrt(ra + soft * soft)
                a = (M * invs ** 3)[:, None] * da
                ph = -M * invs
                if quad:
                    x, y, z = da.unbind(1)
                    qd = torch.stack([Q[:, 0] * x + Q[:, 3] * y + Q[:, 4] * z, Q[:, 3] * x + Q[:, 1] * y + Q[:, 5] * z,
                                      Q[:, 4] * x + Q[:, 5] * y + Q[:, 2] * z], 1)
                    s = (da * qd).sum(1)
                    a += (2.5 * s * inv ** 7)[:, None] * da - (inv ** 5)[:, None] * qd
                    ph -= 0.5 * s * inv ** 5
                acc.index_add_(0, ta, a)
                phi.index_add_(0, ta, ph)
                if w_mlp is not None:
                    band = lev["w"] * inv > THETA_FB
                    tb, cb, hat, M = ta[band], ca[band], -da[band] * inv[band, None], M[band]
                    w = lev["w"]
                    q = Q[band] / (M * w * w)[:, None]
                    A = torch.stack([q[:, 0], q[:, 3], q[:, 4], q[:, 3], q[:, 1], q[:, 5], q[:, 4], q[:, 5], q[:, 2]],
                                    1).reshape(-1, 3, 3)
                    Ah = (A * hat[:, None, :]).sum(2)
                    X = torch.cat([hat, (w * inv[band])[:, None], torch.log10(lev["cnt"][cb].double())[:, None],
                                   (lev["com"][cb] - lev["lo"][cb]) / w - 0.5, (hat * Ah).sum(1, keepdim=True),
                                   Ah.norm(dim=1, keepdim=True), (A * A).sum((1, 2))[:, None],
                                   torch.linalg.det(A)[:, None] if len(A) else A.new_zeros(0, 1)], 1)
                    acc.index_add_(0, tb, (M * inv[band] ** 2)[:, None] * _network(w_mlp, X))
                (t,), c = _expand([t[~ok]], lev["child"][c[~ok]], lev["nchild"][c[~ok]])
    out = torch.empty_like(acc)
    out[T.order] = G * acc
    if not potential:
        return out
    back = torch.empty_like(phi)
    back[T.order] = G * phi
    return out, back


def _images(ng, box, shift):
    return [(gx * box[0], gy * box[1] - gx * shift, gz * box[2]) for gx in range(-ng[0], ng[0] + 1)
            for gy in range(-ng[1], ng[1] + 1) for gz in range(-ng[2], ng[2] + 1)]


def _pairs(x, v, r, ng, box, shift, shear, sweep, h):
    """Colliding pairs (a < b, image of b) in resolution order, with the image's offset and velocity."""
    dev, found = x.device, []
    reach = v[:, 0].abs() * h if sweep else torch.zeros_like(r)
    ext = 2.0 * float((reach + r).max()) * (1.0 + 1e-6)
    if not len(x):
        ext = 0.0
    xs, order = torch.sort(x[:, 0].contiguous())
    g = -1
    for gx in range(-ng[0], ng[0] + 1):
        for gy in range(-ng[1], ng[1] + 1):
            for gz in range(-ng[2], ng[2] + 1):
                g += 1
                o = torch.tensor([gx * box[0], gy * box[1] - gx * shift, gz * box[2]], dtype=x.dtype, device=dev)
                dvy = -gx * shear
                lo = torch.searchsorted(xs, (x[:, 0] - o[0] - ext).contiguous())
                hi = torch.searchsorted(xs, (x[:, 0] - o[0] + ext).contiguous())
                for a0 in range(0, len(x), 1 << 16):
                    a = torch.arange(a0, min(len(x), a0 + (1 << 16)), device=dev)
                    (a,), j = _expand([a], lo[a], (hi - lo)[a])
                    b = order[j]
                    keep = a < b
                    if not sweep:
                        keep &= (x[b, 1] + o[1] - x[a, 1]).abs() < ext
                    a, b = a[keep], b[keep]
                    d = (x[b] + o) - x[a]
                    if sweep:
                        u = v[b] - v[a]
                        u[:, 1] += dvy
                        uu = (u * u).sum(1)
                        tau = torch.where(uu > 0, -(d * u).sum(1) / uu.clamp_min(1e-300), torch.zeros_like(uu)).clamp(-h, h)
                        d = d + u * tau[:, None]
                    hit = (d * d).sum(1) < (r[a] + r[b]) ** 2
                    a, b = a[hit], b[hit]
                    code = (gx + 7) | ((gy + 7) << 4) | ((gz + 7) << 8)
                    found.append(((a << 36) | (b << 12) | code, o.expand(len(a), 3), torch.full_like(d[hit][:, 0], dvy)))
    key = torch.cat([f[0] for f in found])
    key, at = torch.sort(key)
    return key >> 36, (key >> 12) & 0xFFFFFF, torch.cat([f[1] for f in found])[at], torch.cat([f[2] for f in found])[at]


def _resolve(x, v, m, pairs, eps, power):
    """The sorted queue one pair after the other; pairs that share no particle with an earlier one go together."""
    a, b, o, dvy = pairs
    left = torch.arange(len(a), device=x.device)
    n = len(x)
    while len(left):
        first = torch.full((n,), len(a), dtype=torch.long, device=x.device)
        first.scatter_reduce_(0, a[left], left, "amin")
        first.scatter_reduce_(0, b[left], left, "amin")
        ready = (first[a[left]] == left) & (first[b[left]] == left)
        k = left[ready]
        left = left[~ready]
        i, j = a[k], b[k]
        d = (x[j] + o[k]) - x[i]
        u = v[j] - v[i]
        u[:, 1] += dvy[k]
        rv = (d * u).sum(1)
        d2 = (d * d).sum(1)
        e = torch.full_like(rv, eps)
        if power:
            e = ((rv.abs() / torch.sqrt(d2)) / V_C).clamp_min(1e-300).pow(-P_EPS).clamp_max(1.0)
        f = torch.where(rv < 0, (1.0 + e) * rv / (d2 * (m[i] + m[j])), torch.zeros_like(rv))
        v[i] += (f * m[j])[:, None] * d
        v[j] -= (f * m[i])[:, None] * d


def _drift(cfg, x, v, tau):
    if cfg.integrator == rb.RB_INT_LEAPFROG:
        return x + v * tau, v
    O = cfg.omega
    ph = O * tau
    c, s = math.cos(ph), math.sin(ph)
    X, Y, Z = x.unbind(1)
    U, V, W = v.unbind(1)
    # the force-free solution of Hill's equations over tau
    nx = torch.stack([(4 - 3 * c) * X + s / O * U + 2 / O * (1 - c) * V,
                      Y + (6 * (s - ph) * X - 2 / O * (1 - c) * U + (4 * s - 3 * ph) / O * V), c * Z + s / O * W], 1)
    nv = torch.stack([3 * O * s * X + c * U + 2 * s * V, 6 * O * (c - 1) * X - 2 * s * U + (4 * c - 3) * V,
                      -O * s * Z + c * W], 1)
    return nx, nv


def _wrap(cfg, box, x, v, shift, shear):
    for sign in (1.0, -1.0):
        out = x[:, 0] >= 0.5 * box[0] if sign > 0 else x[:, 0] < -0.5 * box[0]
        x[out, 0] -= sign * box[0]
        x[out, 1] += sign * shift
        v[out, 1] += sign * shear
    for k in ((1, 2) if cfg.z_periodic else (1,)):
        # one box length at a time: the azimuthal shear carries particles of a long ring several boxes on
        while bool((up := x[:, k] >= 0.5 * box[k]).any()):
            x[up, k] -= box[k]
        while bool((down := x[:, k] < -0.5 * box[k]).any()):
            x[down, k] += box[k]


def _too_long(case):
    """Cases whose 64-bit result would take over about 20 seconds."""
    if case["kind"] == "ensemble":
        return case["boxes"] * case["steps"] > 130
    n, steps = case["n"], case.get("steps", 1)
    if case["kind"] == "ring" or not case.get("gravity", True):
        return n * steps > 1_300_000
    return n * steps / case["theta"] ** 2 > (500_000 if case["kind"] == "plummer" else 1_700_000)


def exact(case, seed):
    if case["kind"] == "train" or _too_long(case):
        return None   # training: the rows' order comes from the library's own shuffle
    dev, got, states = _device(), {}, []
    w_mlp = _weights(seed) if case.get("walk") == "learned" else None
    power = case.get("law") == "power"
    boxes = _boxes(case, seed)
    cfg = rb.make_config(**_config(case, seed, boxes[0][0]))
    for b, (box, P) in enumerate(boxes):
        x = torch.tensor(np.stack([P.x, P.y, P.z], 1), device=dev)
        v = torch.tensor(np.stack([P.vx, P.vy, P.vz], 1), device=dev)
        m, r = torch.tensor(P.m, device=dev), torch.tensor(P.r, device=dev)
        src = m.clone()
        if case.get("tracers"):
            src[P.n // 2:] = 0.0
        if case["kind"] == "plummer":
            return dict(a=_forces(x, src, box, [(0.0, 0.0, 0.0)], cfg.G, cfg.theta, cfg.softening, True).cpu())
        ng = tuple(cfg.nghost)
        sheared = cfg.boundary == rb.RB_BC_SHEAR
        shear = 1.5 * cfg.omega * box[0] if sheared else 0.0
        h = 0.5 * cfg.dt

        def shift(k):
            return math.fmod(shear * (cfg.t0 + k * h), box[1]) if sheared else 0.0

        for s in range(case["steps"]):
            x, v = _drift(cfg, x, v, h)
            _wrap(cfg, box, x, v, shift(2 * s + 1), shear)
            if cfg.gravity:
                v = v + cfg.dt * _forces(x, src, box, _images(ng, box, shift(2 * s + 1)), cfg.G, cfg.theta, cfg.softening,
                                         cfg.quadrupole, w_mlp)
            x, v = _drift(cfg, x, v, h)
            _wrap(cfg, box, x, v, shift(2 * s + 2), shear)
            pairs = _pairs(x, v, r, ng, box, shift(2 * s + 2), shear, cfg.collisions == rb.RB_COLL_SWEEP, h)
            _resolve(x, v, m, pairs, cfg.eps_restitution, power)
        states.append(torch.cat([x, v], 1))
        if case.get("energy"):
            _, phi = _forces(x, src, box, _images(ng, box, shift(2 * case["steps"])), cfg.G, cfg.theta, cfg.softening,
                             cfg.quadrupole, None, True)
            K = float((0.5 * m * (v * v).sum(1)).sum())
            U = float((m * (0.5 * cfg.omega ** 2 * x[:, 2] ** 2 - 1.5 * cfg.omega ** 2 * x[:, 0] ** 2)).sum())
            got["terms"] = [K, U, float(0.5 * (m * phi).sum())]
            got["momentum"] = (m[:, None] * v).sum(0).cpu()
    got.update(zip(STATE, torch.cat(states).cpu().unbind(1)))
    return got
