"""Timed cases of the assembly library: what a simulation or an optimisation asks of it per frame.

A case is a dict of plain values.  ``listed()`` names the standing ones, ``draw(rng)`` gives one
more of the same ranges, ``prepare(case, seed)`` builds what a program has in hand before the
call, ``run(state)`` makes one pass through the public entry points, ``work(case)`` counts what
such a pass cannot do without and ``exact(case, seed)`` gives the outputs in plain 64-bit torch.

Meshes (the shapes of the repository's workloads, built here with array operations only):

* ``block``     n^3 hexes cut into 6 tetrahedra each, jittered nodes;
* ``fracture``  a block whose tetrahedra along the faces of a Voronoi partition have preallocated
                split copies (inactive at start), swapped in when an interface breaks;
* ``refine``    a block whose every tetrahedron has its 8 preallocated red-refinement children,
                a refined ball moving through it;
* ``batch``     many independent blocks in one context.

The connectivity follows from the case; node positions, materials, masks, edits, loads and
gradients are drawn from the seed.  Frames of a stream run forwards and then backwards
(fracture, then merge), so a pass can be repeated for as long as wanted.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_2605_11673_gb300 as P
from paper_2605_11673_gb300 import autograd as G

FRAMES = 4            # frames of a stream before it turns back
RHO, DT = 1000.0, 1e-3
PAIRS = [(a, b) for a in range(4) for b in range(a, 4)]


# ----------------------------------------------------------------------------------------
# Cases
# ----------------------------------------------------------------------------------------

def listed():
    return [
        # an interactive toy: the smallest mesh and a few dozen edits, all launch latency
        dict(name="frame_small", kind="frame", mesh="block", n=6, rate=0.02, policy=0, graph=True, eps=0.0),
        # the headline: interfaces of a pre-fractured block break, CUDA-graph mode
        dict(name="frame_fracture", kind="frame", mesh="fracture", n=40, rate=0.0, policy=0, graph=True, eps=0.0),
        # adaptive refinement: thousands of tetrahedra a frame, eps on the diagonal, plain launches
        dict(name="frame_refine", kind="frame", mesh="refine", n=24, rate=0.3, policy=0, graph=False, eps=0.5),
        # 48 scenes of a training batch streamed together, large frames
        dict(name="frame_batch", kind="frame", mesh="batch", n=48, rate=0.02, policy=0, graph=True, eps=0.0),
        # the exact additive policy on the headline mesh
        dict(name="frame_fixed", kind="frame", mesh="fracture", n=40, rate=0.0, policy=1, graph=True, eps=0.0),
        # a scene reset: a new active mask from host memory, every value rebuilt
        dict(name="rebuild_mask", kind="rebuild", mesh="fracture", n=40, rate=0.0, policy=0, source="host", eps=0.0),
        # the rebuild alone on a mostly inactive superset of 1.46 M tetrahedra (the largest)
        dict(name="refold_refine", kind="rebuild", mesh="refine", n=30, rate=0.15, policy=0, source="refold", eps=0.0),
        # one step of material and shape optimisation: assembly and its adjoint, small and large
        dict(name="assemble_grad", kind="assemble_grad", mesh="block", n=20),
        dict(name="assemble_grad_large", kind="assemble_grad", mesh="block", n=40),
        # the consumer of that step: a static solve and its adjoint
        dict(name="solve_grad", kind="solve_grad", mesh="block", n=20),
        # a frame of the implicit-Euler loop: edits, lumped mass, CG; the take is played again from
        # its saved state after 8 frames
        dict(name="dynamics", kind="dynamics", mesh="fracture", n=40),
        # a frame of the graph-Laplacian operator: edits, then its solve
        dict(name="proxy_frame", kind="proxy", mesh="fracture", n=40),
    ]


def _spread(rng, lo, hi):
    """Whole number in [lo, hi], uniform over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "rebuild", "rebuild", "assemble_grad", "solve_grad", "dynamics", "proxy"])
    if kind in ("frame", "rebuild"):
        mesh = rng.choice(["block", "fracture", "refine", "batch"])
        c = dict(kind=kind, mesh=mesh, policy=rng.choice([0, 0, 0, 1]), eps=rng.choice([0.0, 0.5]))
        c["n"] = {"block": (4, 40), "fracture": (8, 40), "refine": (5, 28), "batch": (2, 48)}[mesh]
        c["n"] = _spread(rng, *c["n"])
        # block, batch: share of the tetrahedra edited a frame; refine: radius of the ball
        c["rate"] = round(rng.uniform(0.1, 0.4) if mesh == "refine" else math.exp(rng.uniform(math.log(0.002), math.log(0.05))), 4)
        if kind == "frame":
            c["graph"] = rng.random() < 0.7
        else:
            c["source"] = rng.choice(["host", "device", "refold"])
        return c
    if kind in ("assemble_grad", "solve_grad"):
        return dict(kind=kind, mesh="block", n=_spread(rng, 5, 40 if kind == "assemble_grad" else 20))
    return dict(kind=kind, mesh="fracture", n=_spread(rng, 8, 40))


# ----------------------------------------------------------------------------------------
# Meshes and streams (numpy; the searches over all tetrahedra in torch)
# ----------------------------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _block(n, jitter, rng):
    """n^3 hexes of the unit cube, each cut into 6 tetrahedra along its (0,0,0)-(1,1,1) diagonal,
    positively oriented; nodes jittered by +-jitter h."""
    h, m = 1.0 / n, n + 1
    g = np.arange(m)
    X = np.stack([np.tile(g, m * m), np.tile(np.repeat(g, m), m), np.repeat(g, m * m)], 1) * h
    X += rng.uniform(-jitter * h, jitter * h, X.shape)
    c = np.arange(n)
    base = (c[None, None, :] + m * (c[None, :, None] + m * c[:, None, None])).reshape(-1)
    step = (1, m, m * m)
    tets = np.empty((n ** 3, 6, 4), np.int32)
    for k, p in enumerate(itertools.permutations(range(3))):
        odd = sum(p[i] > p[j] for i in range(3) for j in range(i + 1, 3)) % 2
        v = [base, base + step[p[0]], base + step[p[0]] + step[p[1]], base + sum(step)]
        if odd:
            v[2], v[3] = v[3], v[2]
        for a in range(4):
            tets[:, k, a] = v[a]
    return X, tets.reshape(-1, 4)


def _edits(off=(), on=(), swap=None):
    off, on = np.asarray(off, np.int32), np.asarray(on, np.int32)
    e = [np.stack([np.zeros_like(off), off, np.full_like(off, -1)], 1),
         np.stack([np.ones_like(on), on, np.full_like(on, -1)], 1)]
    if swap is not None:
        a, b = (np.asarray(x, np.int32) for x in swap)
        e.append(np.stack([np.full_like(a, 2), a, b], 1))
    return np.ascontiguousarray(np.concatenate(e))


def _back(e):
    """The frame that undoes a frame."""
    r = e.copy()
    r[:, 0] = np.where(e[:, 0] == 2, 2, 1 - e[:, 0])
    sw = e[:, 0] == 2
    r[sw, 1], r[sw, 2] = e[sw, 2], e[sw, 1]
    return r


def _after(mask, e):
    m = mask.copy()
    m[e[e[:, 0] != 1, 1]] = 0
    m[e[e[:, 0] == 1, 1]] = 1
    m[e[e[:, 0] == 2, 2]] = 1
    return m


def _random_stream(T, rate, rng):
    """All but a few tetrahedra active; each frame deactivates `rate` of them and reactivates a
    quarter as many of the inactive ones."""
    k = max(1, int(round(rate * T)))
    mask = np.ones(T, np.uint8)
    order = rng.permutation(T)
    ina = order[:min(k, T // 4)]
    mask[ina] = 0
    frames, m = [], mask.copy()
    for _ in range(FRAMES):
        act, dead = np.flatnonzero(m), np.flatnonzero(m == 0)
        e = _edits(off=rng.choice(act, min(k, act.size), replace=False),
                   on=rng.choice(dead, min(max(1, k // 4), dead.size), replace=False))
        frames.append(e)
        m = _after(m, e)
    return mask, frames


def _fracture(n, rng):
    """Voronoi partition of the block (64 cells at n = 40, fewer on a smaller one); every
    tetrahedron with a node on a cell face gets a copy whose face nodes are private to its cell.
    Each frame breaks 3 cell-cell interfaces: the tetrahedra of either cell that touch both are
    swapped for their copies.  Which interfaces break, and in which order, comes from the seed."""
    X, tets = _block(n, 0.15, rng)
    T0, n0 = len(tets), len(X)
    fixed = np.random.default_rng([2, n])
    sites = torch.as_tensor(fixed.uniform(0, 1, (max(3, n * n // 25), 3)), device=_device())
    lattice = torch.as_tensor(_block(n, 0.0, fixed)[0], device=_device())
    cen = lattice[torch.as_tensor(tets, device=_device()).long()].mean(1)
    cell = torch.cat([((c[:, None] - sites) ** 2).sum(-1).argmin(1) for c in cen.split(1 << 17)]).cpu().numpy()
    S = len(sites)
    key = tets.astype(np.int64) * S + cell[:, None]            # (node, cell) of every corner
    uk = torch.unique(torch.as_tensor(key.reshape(-1), device=_device())).cpu().numpy()
    face = np.bincount(uk // S, minlength=n0) >= 2             # nodes on a cell face
    dup = uk[face[uk // S]]                                    # their (node, cell) pairs
    orig = np.flatnonzero(face[tets].any(1))
    ck = key[orig]
    copies = np.where(face[tets[orig]], n0 + np.searchsorted(dup, ck), tets[orig]).astype(np.int32)
    copy_of = np.full(T0, -1, np.int64)
    copy_of[orig] = T0 + np.arange(orig.size)
    mask = np.concatenate([np.ones(T0, np.uint8), np.zeros(orig.size, np.uint8)])
    in_cell = [np.flatnonzero(cell[orig] == s) for s in range(S)]
    nodes_of = [dup[dup % S == s] // S for s in range(S)]
    frames, swapped = [], np.zeros(T0, bool)
    for _ in range(FRAMES):
        sel = []
        for _ in range(3):
            a = int(rng.integers(S))
            near = [b for b in range(S) if b != a and np.intersect1d(nodes_of[a], nodes_of[b], True).size]
            b = near[int(rng.integers(len(near)))]
            flag = np.zeros(n0, bool)
            flag[np.intersect1d(nodes_of[a], nodes_of[b], True)] = True
            t = orig[np.concatenate([in_cell[a], in_cell[b]])]
            t = t[flag[tets[t]].any(1) & ~swapped[t]]
            swapped[t] = True
            sel.append(t)
        sel = np.concatenate(sel)
        rng.shuffle(sel)
        frames.append(_edits(swap=(sel, copy_of[sel])))
    X = np.concatenate([X, X[dup // S]])
    return X, np.concatenate([tets, copies]), mask, frames


def _refine(n, radius, rng):
    """Every tetrahedron of the block has 8 preallocated children; a ball of the given radius
    moves through it, a parent whose centroid it covers is replaced by its children.  A frame
    moves the ball by 4% of the cube."""
    X, tets = _block(n, 0.0, rng)
    T0, n0 = len(tets), len(X)
    e = np.sort(np.concatenate([tets[:, [a, b]] for a, b in itertools.combinations(range(4), 2)]), 1).astype(np.int64)
    key = torch.unique(torch.as_tensor(e[:, 0] * n0 + e[:, 1], device=_device())).cpu().numpy()
    v = [tets[:, k].astype(np.int64) for k in range(4)]

    def mid(a, b):
        lo, hi = np.minimum(v[a], v[b]), np.maximum(v[a], v[b])
        return n0 + np.searchsorted(key, lo * n0 + hi)

    m01, m02, m03, m12, m13, m23 = (mid(a, b) for a, b in itertools.combinations(range(4), 2))
    kids = [(v[0], m01, m02, m03), (m01, v[1], m12, m13), (m02, m12, v[2], m23), (m03, m13, m23, v[3]),
            (m01, m02, m03, m13), (m01, m02, m12, m13), (m02, m03, m13, m23), (m02, m12, m13, m23)]
    ch = np.stack([np.stack(k, -1) for k in kids], 1).reshape(-1, 4).astype(np.int32)
    X = np.concatenate([X, 0.5 * (X[key // n0] + X[key % n0])])
    d = X[ch[:, 1:]] - X[ch[:, :1]]
    neg = np.einsum("ij,ij->i", d[:, 0], np.cross(d[:, 1], d[:, 2])) < 0
    ch[neg, 2], ch[neg, 3] = ch[neg, 3].copy(), ch[neg, 2].copy()
    cen = X[tets].mean(1)
    p = rng.uniform(0.3, 0.7, 3)
    u = rng.standard_normal(3)
    u *= 0.04 / np.linalg.norm(u)
    ins = [((cen - (p + k * u)) ** 2).sum(1) < radius * radius for k in range(FRAMES + 1)]
    mask = np.concatenate([(~ins[0]).astype(np.uint8), np.repeat(ins[0], 8).astype(np.uint8)])
    frames, kid = [], T0 + np.arange(8)
    for r0, r1 in zip(ins, ins[1:]):
        up, down = np.flatnonzero(r1 & ~r0), np.flatnonzero(r0 & ~r1)
        frames.append(_edits(off=np.concatenate([up, (8 * down[:, None] + kid).reshape(-1)]),
                             on=np.concatenate([(8 * up[:, None] + kid).reshape(-1), down])))
    return X, np.concatenate([tets, ch]), mask, frames


def _materials(T, rng):
    return 1e5 * np.exp(0.3 * rng.standard_normal(T)), rng.uniform(0.2, 0.4, T)


def _scene(case, seed):
    """Host arrays of a case's mesh(es): a list of (X, tets, E, nu, mask, frames)."""
    rng = np.random.default_rng(seed)
    mesh = case["mesh"]
    if mesh == "batch":
        out = []
        fixed = np.random.default_rng([4, case["n"]])
        for t in np.exp(fixed.uniform(math.log(2e3), math.log(5e4), case["n"])):
            X, tets = _block(max(1, int(round((t / 6) ** (1 / 3)))), 0.15, rng)
            out.append((X, tets, *_materials(len(tets), rng), *_random_stream(len(tets), case["rate"], rng)))
        return out
    if mesh == "fracture":
        X, tets, mask, frames = _fracture(case["n"], rng)
    elif mesh == "refine":
        X, tets, mask, frames = _refine(case["n"], case["rate"], rng)
    else:
        X, tets = _block(case["n"], 0.15, rng)
        mask, frames = _random_stream(len(tets), case.get("rate", 0.02), rng)
    return [(X, tets, *_materials(len(tets), rng), mask, frames)]


def _cracked(n):
    """Active mask of a block with a half-through crack: one layer of hexes open over x < 1/2."""
    act = np.ones((n, n, n), np.uint8)
    act[n // 2, :, : n // 2] = 0
    return np.repeat(act.reshape(-1), 6)


def _supports(X):
    """(clamped nodes, load): the bottom is clamped, a downward load is spread over the top."""
    h = 0.5 / max(1, round(len(X) ** (1 / 3)))
    top = X[:, 2] > X[:, 2].max() - h
    f = np.zeros_like(X)
    f[top, 2] = -1e3 / top.sum()
    return X[:, 2] < X[:, 2].min() + h, f.reshape(-1)


# ----------------------------------------------------------------------------------------
# prepare, run
# ----------------------------------------------------------------------------------------

def _cuda(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _cycle(per_scene):
    """The stream forwards, then backwards."""
    return per_scene + [_back(e) for e in reversed(per_scene)]


def prepare(case, seed):
    kind, sc = case["kind"], _scene(case, seed)
    rng = np.random.default_rng([seed, 1])
    X, tets, E, nu, mask, frames = sc[0]
    s = {"kind": kind, "k": 0}
    if kind == "proxy":
        asm = P.ProxyAssembler(len(X), tets, eps=1e-2)
        asm.full_rebuild(mask)
        s.update(frames=_cycle(frames), b=_cuda(rng.standard_normal(len(X))))
        s.update(free=torch.ones(len(X), dtype=torch.uint8, device="cuda"), x=None, state=asm.state())
    elif case["mesh"] == "batch":
        asm = P.BatchAssembler([q[:4] for q in sc], eps=case["eps"])
        mask = np.concatenate([q[4] for q in sc])
        asm.full_rebuild(mask)
        streams = [_cycle(q[5]) for q in sc]
        s["frames"] = [list(f) for f in zip(*streams)]
        off = np.cumsum([0] + [len(q[1]) for q in sc])
        frames = [np.concatenate([e + np.where(e < 0, 0, o) * np.array([0, 1, 1], np.int32) for e, o in zip(f, off)])
                  for f in s["frames"]]
    else:
        asm = P.Assembler(X, tets, E, nu, eps=case.get("eps", 0.0))
        if kind in ("assemble_grad", "solve_grad"):
            mask = _cracked(case["n"])
        asm.full_rebuild(mask)
        s["frames"] = _cycle(frames)
    if case.get("policy"):
        asm.set_policy(P.STA_POLICY_FIXED)
    if kind == "rebuild":
        masks, m = [], mask
        for e in (frames if case["mesh"] != "batch" else frames[:FRAMES]):
            m = _after(m, e)
            masks.append(m)
        asm.full_rebuild(masks[-1])
        if case["source"] == "device":
            masks = [_cuda(m, torch.uint8) for m in masks]
        s.update(masks=masks, source=case["source"])
    if kind == "assemble_grad":
        s.update(E=_cuda(E).requires_grad_(), nu=_cuda(nu).requires_grad_(), X=_cuda(X).requires_grad_())
        s["g"] = _cuda(rng.standard_normal(asm.nnz))
    if kind == "solve_grad":
        clamped, f = _supports(X)
        act = np.zeros(len(X), bool)
        act[np.unique(tets[mask != 0])] = True
        s.update(free=_cuda(np.repeat(act & ~clamped, 3), torch.bool), f=_cuda(f).requires_grad_())
        s["val"] = asm.values().clone().requires_grad_()
    if kind == "dynamics":
        clamped, f = _supports(X)
        asm.dyn_setup(RHO, DT, f, clamped)
        s["state"] = asm.dyn_state()
        s["rest"] = np.zeros(3 * len(X))
    if case.get("graph", kind in ("dynamics", "proxy")):
        largest = max(int(len(e) + (e[:, 0] == 2).sum()) for f in s["frames"] for e in [f if not isinstance(f, list) else np.concatenate(f)])
        asm.graph_enable(largest)
    s.update(asm=asm, val_view=asm.values())
    return s


def run(s):
    asm, kind = s["asm"], s["kind"]
    if kind == "assemble_grad":
        v = G.Assemble.apply(s["E"], s["nu"], s["X"], asm)
        return [v.detach(), *torch.autograd.grad(v, (s["E"], s["nu"], s["X"]), s["g"])]
    if kind == "solve_grad":
        u = G.Solve.apply(s["val"], s["f"], asm, s["free"])
        return [u.detach(), *torch.autograd.grad(u, (s["val"], s["f"]), s["f"].detach())]
    k = s["k"]
    s["k"] = k + 1
    if kind == "rebuild":
        if s["source"] == "refold":
            asm.refold()
        else:
            asm.full_rebuild(s["masks"][k % len(s["masks"])])
        return [s["val_view"]]
    if kind == "dynamics" and k and k % len(s["frames"]) == 0:
        asm.dyn_set_state(s["rest"], s["rest"])
    asm.apply_edits(s["frames"][k % len(s["frames"])])
    if kind == "dynamics":
        asm.dyn_step()
        return [s["val_view"], *s["state"]]
    if kind == "proxy":
        s["x"], _, _ = P.sta_solve(asm.h, s["b"], s["free"], x0=s["x"])
        return [s["val_view"], *s["state"], s["x"]]
    return [s["val_view"]]


# ----------------------------------------------------------------------------------------
# work, exact
# ----------------------------------------------------------------------------------------

class _Pattern:
    """Superset pattern of a mesh in torch: node-pair blocks in CSR order."""

    def __init__(self, n, tets):
        self.n, self.dev = n, _device()
        self.t = torch.as_tensor(tets, device=self.dev).long()
        key = torch.unique(torch.cat([self.t[:, a] * n + self.t[:, b] for a in range(4) for b in range(4)]))
        self.key, self.row = key, key // n
        self.deg = torch.bincount(self.row, minlength=n)
        self.start = torch.cumsum(self.deg, 0) - self.deg
        self.nblocks = key.numel()

    def entries(self, t):
        """CSR index of every entry of the 12x12 matrices of tetrahedra t: (m, 12, 12)."""
        v = self.t[t]
        g = torch.searchsorted(self.key, (v[:, :, None] * self.n + v[:, None, :]).reshape(-1)).view(-1, 4, 4)
        s, d = self.start[v][:, :, None], self.deg[v][:, :, None]
        i = torch.arange(3, device=self.dev)
        idx = (9 * s + 3 * (g - s))[:, :, None, :, None] + (3 * d)[:, :, None, :, None] * i[:, None, None] + i
        return idx.reshape(-1, 12, 12)

    def csr(self, val):
        """(3n x 3n) sparse matrix of values in the context's order."""
        rows = 3 * self.n
        rp = torch.zeros(rows + 1, dtype=torch.long, device=self.dev)
        rp[1:] = torch.cumsum((3 * self.deg).repeat_interleave(3), 0)
        a = torch.arange(rows, device=self.dev).repeat_interleave((3 * self.deg).repeat_interleave(3))
        off = torch.arange(val.numel(), device=self.dev) - rp[a]
        col = 3 * (self.key % self.n)[self.start[a // 3] + off // 3] + off % 3
        return torch.sparse_csr_tensor(rp, col, val, (rows, rows)), a, col


def _elements(X, t, E, nu):
    """K = V B^T D B of linear tetrahedra, (m, 12, 12), and their volumes."""
    x = X[t]
    d = x[:, 1:] - x[:, :1]
    vol = torch.linalg.det(d) / 6
    g = torch.linalg.inv(d).transpose(1, 2)
    g = torch.cat([-g.sum(1, keepdim=True), g], 1)
    lam, mu = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    gg = torch.einsum("tai,tbi->tab", g, g)
    I = torch.eye(3, dtype=X.dtype, device=X.device)
    K = (lam[:, None, None, None, None] * torch.einsum("tai,tbj->taibj", g, g)
         + mu[:, None, None, None, None] * (torch.einsum("taj,tbi->taibj", g, g) + torch.einsum("tab,ij->taibj", gg, I)))
    return (vol[:, None, None, None, None] * K).reshape(-1, 12, 12), vol


def _assembled(pat, X, E, nu, mask, eps):
    X, E, nu = (torch.as_tensor(a, device=pat.dev) for a in (X, E, nu))
    val = torch.zeros(9 * pat.nblocks, dtype=torch.float64, device=pat.dev)
    for t in torch.nonzero(torch.as_tensor(mask, device=pat.dev))[:, 0].split(1 << 17):
        K, _ = _elements(X, pat.t[t], E[t], nu[t])
        val.index_add_(0, pat.entries(t).reshape(-1), K.reshape(-1))
    if eps:
        a = torch.arange(pat.n, device=pat.dev)[pat.deg > 0]
        g = torch.searchsorted(pat.key, a * pat.n + a) - pat.start[a]
        for i in range(3):
            val[9 * pat.start[a] + 3 * i * pat.deg[a] + 3 * g + i] += eps
    return val


def _solve(A, diag, b, free, x=None, tol=1e-15, most=6000):
    """Jacobi-PCG in plain torch on the free rows, restarted once from its own residual."""
    fr = free.to(b.dtype)
    inv = torch.where(diag != 0, fr / torch.where(diag != 0, diag, torch.ones_like(diag)), torch.zeros_like(diag))
    x = torch.zeros_like(b) if x is None else x * fr
    bb = float(torch.linalg.norm(b * fr))
    for _ in range(2):
        r = fr * (b - A(x))
        z = inv * r
        p, rz = z.clone(), z @ r
        for k in range(most):
            if k % 25 == 0 and not float(torch.linalg.norm(r)) > tol * bb:
                break
            q = fr * A(p)
            al = rz / (p @ q)
            x = x + al * p
            r = r - al * q
            z = inv * r
            rn = z @ r
            p = z + (rn / rz) * p
            rz = rn
    return x


def exact(case, seed):
    kind, sc = case["kind"], _scene(case, seed)
    rng = np.random.default_rng([seed, 1])
    X, tets, E, nu, mask, frames = sc[0]
    eps = case.get("eps", 0.0)
    if kind in ("frame", "rebuild"):
        out = []
        for X, tets, E, nu, mask, frames in sc:
            if kind == "rebuild" and case["source"] == "refold":
                for e in frames:
                    mask = _after(mask, e)
            else:
                mask = _after(mask, frames[0])
            out.append(_assembled(_Pattern(len(X), tets), X, E, nu, mask, eps))
        return [torch.cat(out)]
    pat = _Pattern(len(X), tets)
    dev = pat.dev
    if kind == "assemble_grad":
        mask = _cracked(case["n"])
        g = torch.as_tensor(rng.standard_normal(9 * pat.nblocks), device=dev)
        leaf = [torch.as_tensor(a, device=dev).requires_grad_() for a in (E, nu, X)]
        grads = [torch.zeros_like(a) for a in leaf]
        for t in torch.nonzero(torch.as_tensor(mask, device=dev))[:, 0].split(1 << 16):
            K, _ = _elements(leaf[2], pat.t[t], leaf[0][t], leaf[1][t])
            for a, d in zip(grads, torch.autograd.grad((K * g[pat.entries(t)]).sum(), leaf)):
                a += d
        return [_assembled(pat, X, E, nu, mask, 0.0), *grads]
    if kind == "proxy":
        mask = _after(mask, frames[0])
        t = pat.t[torch.as_tensor(mask != 0, device=dev)]
        lo_hi = [(torch.minimum(t[:, a], t[:, b]), torch.maximum(t[:, a], t[:, b])) for a, b in PAIRS if a != b]
        g = torch.searchsorted(pat.key, torch.cat([lo * pat.n + hi for lo, hi in lo_hi]))
        mult = torch.bincount(g, minlength=pat.nblocks)
        col = pat.key % pat.n
        up = torch.searchsorted(pat.key, torch.minimum(pat.row, col) * pat.n + torch.maximum(pat.row, col))
        on = (mult[up] > 0).double()
        deg = torch.zeros(pat.n, dtype=torch.float64, device=dev).index_add_(0, pat.row, on)
        val = torch.where(pat.row == col, deg[pat.row] + 1e-2, -on)
        b = torch.as_tensor(rng.standard_normal(pat.n), device=dev)
        rp = torch.cat([torch.zeros(1, dtype=torch.long, device=dev), torch.cumsum(pat.deg, 0)])
        A = torch.sparse_csr_tensor(rp, col, val, (pat.n, pat.n))
        free = pat.deg > 0
        x = _solve(lambda v: A @ v, torch.where(free, deg + 1e-2, torch.zeros_like(deg)), b, free)
        return [val, None, None, x]
    if kind == "solve_grad":
        mask = _cracked(case["n"])
        val = _assembled(pat, X, E, nu, mask, 0.0)
        clamped, f = _supports(X)
        act = np.zeros(len(X), bool)
        act[np.unique(tets[mask != 0])] = True
        free = torch.as_tensor(np.repeat(act & ~clamped, 3), device=dev)
        A, row, col = pat.csr(val)
        diag = torch.zeros(3 * pat.n, dtype=torch.float64, device=dev).index_add_(0, row, torch.where(row == col, val, torch.zeros_like(val)))
        f = torch.as_tensor(f, device=dev)
        u = _solve(lambda v: A @ v, diag, f, free)   # lam = u: the upstream gradient is f
        uf = u * free
        return [u, -uf[row] * uf[col], uf]
    # dynamics, the first step from rest
    mask = _after(mask, frames[0])
    val = _assembled(pat, X, E, nu, mask, 0.0)
    clamped, f = _supports(X)
    t = pat.t[torch.as_tensor(mask != 0, device=dev)]
    x = torch.as_tensor(X, device=dev)[t]
    q = RHO * torch.linalg.det(x[:, 1:] - x[:, :1]) / 24
    mass = torch.zeros(pat.n, dtype=torch.float64, device=dev).index_add_(0, t.reshape(-1), q.repeat_interleave(4))
    A, row, col = pat.csr(val)
    diag = torch.zeros(3 * pat.n, dtype=torch.float64, device=dev).index_add_(0, row, torch.where(row == col, val, torch.zeros_like(val)))
    m3, h2 = mass.repeat_interleave(3), DT * DT
    free = torch.as_tensor(np.repeat(~clamped, 3), device=dev) & (m3 > 0)
    u = _solve(lambda v: m3 * v + h2 * (A @ v), m3 + h2 * diag, h2 * torch.as_tensor(f, device=dev), free)
    return [val, u, u / DT, mass]


def work(case):
    """Bytes: each input read once, each output written once; flops: the additions and
    multiplications of the sums asked for.  A re-folded frame reads the active contributions of
    the entries it writes; a solve is charged one application of its matrix (how many it takes
    is the solver's own doing)."""
    kind, total = case["kind"], {"bytes": 0, "flops": 0}

    def add(b, f):
        total["bytes"] += int(b)
        total["flops"] += int(f)

    for X, tets, E, nu, mask, frames in _scene(case, 0):
        n, T = len(X), len(tets)
        t = torch.as_tensor(tets, device=_device()).long()
        pairs = torch.stack([torch.minimum(t[:, a], t[:, b]) * n + torch.maximum(t[:, a], t[:, b]) for a, b in PAIRS], 1)
        key = torch.unique(pairs)
        ndiag = int((key // n == key % n).sum())
        nnz = 9 * (2 * key.numel() - ndiag)
        if kind in ("assemble_grad", "solve_grad"):
            mask = _cracked(case["n"])
        act = int(mask.sum())
        if kind == "rebuild":
            add((T if case["source"] != "refold" else 0) + 624 * act + 8 * nnz, 78 * act)
        elif kind == "assemble_grad":  # forward: inputs, values; backward: inputs, gradient, gradients
            add(2 * (16 * T + 16 * act + 24 * n) + T + 16 * nnz + 16 * T + 24 * n, (307 + 78 + 550) * act)
        elif kind == "solve_grad":     # two solves and the outer product
            add(2 * (8 * nnz + 24 * n) + 8 * nnz + 5 * 24 * n, 2 * 2 * nnz + nnz)
        else:
            e = frames[0]
            ids = np.concatenate([e[:, 1], e[e[:, 0] == 2, 2]])
            touched = torch.unique(pairs[torch.as_tensor(ids, device=t.device).long()])
            dg = touched // n == touched % n
            entries = int(9 * dg.sum() + 18 * (~dg).sum())
            if kind == "proxy":
                add(12 * len(e) + 40 * ids.size + 12 * (entries // 9) + 8 * (nnz // 9) + 4 * (nnz // 9) + 16 * n, 2 * (nnz // 9))
                continue
            if case.get("policy"):
                add(12 * len(e) + 624 * ids.size + 16 * entries, 78 * ids.size)
            else:
                on = pairs[torch.as_tensor(_after(mask, e) != 0, device=t.device)]
                at = torch.searchsorted(touched, on).clamp_(max=touched.numel() - 1)
                hit = touched[at] == on
                dcol = torch.as_tensor([a == b for a, b in PAIRS], device=t.device)
                ops = int(6 * (hit & dcol).sum() + 9 * (hit & ~dcol).sum())
                add(12 * len(e) + 8 * ops + 8 * entries, ops)
            if kind == "dynamics":
                add(8 * nnz + 24 * n * 5 + 8 * n, 2 * nnz)
    return total
