"""The work a user of this framework has it do, as cases that can be timed and compared: inputs, one pass
through the public entry points, and the same results from plain torch in 64 bits.

A case names a `kind` of pass:
  trip   bin the particles, project them onto the mesh (P2M) and back (M2P): one step of a simulation
  m2p    mesh -> particles alone, at positions in hand
  loop   steps of the projection loop: M2P, midpoint move, re-binning, P2M
  grad   P2M (and M2P) with the gradients of a mismatch loss by values and positions
  batch  round trips of many uneven problems at once
Meshes have n x n nodes (image row and column included) and particle sets m x m particles, on a lattice
jittered by `jitter` spacings or (`jitter` None) uniformly random."""
import math
import random

import torch

import paper_1610_05266_gb300 as P
from paper_1610_05266_gb300 import autograd as PA

DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
SOLVES = {"f64": P.PFEM_SOLVE_F64, "f32": P.PFEM_SOLVE_F32, "refined": P.PFEM_SOLVE_F32_REFINED,
          "refined_ff": P.PFEM_SOLVE_F32_REFINED_FF}
SHAPES = {"linear": P.PFEM_SHAPE_LINEAR, "quadratic": P.PFEM_SHAPE_QUADRATIC}
DEVICE = "cuda"


def listed():
    return [
        # the smallest configuration: a coarse mesh in the paper's own precision, launches and latency
        trip("tiny_f64", 33, 64, 3, "f64", "f64"),
        # an odd, ragged mid-size problem with three fields
        trip("ragged_f32", 138, 271, 3, "f32", "refined"),
        # the headline configuration: four fields at four particles per node
        trip("large_f32", 1025, 2048, 4, "f32", "refined"),
        # the precision study's sizes: one density field with BF16 storage, the widest arrays
        trip("wide_bf16", 4097, 8192, 1, "bf16", "refined"),
        # the paper's precision on a production mesh
        trip("large_f64", 513, 1024, 3, "f64", "f64"),
        # particles that have lost their lattice: sparse spots, long stars, ill-conditioned systems
        trip("random_f32", 513, 1024, 3, "f32", "refined", jitter=None),
        # projFEM6: linear shape functions, six particles per node
        trip("fe_six_f32", 513, 1254, 3, "f32", "f32", shape="linear", m2p="linear"),
        # mesh -> particles with the mesh's quadratically consistent shape functions
        {"name": "m2p_quadratic", "kind": "m2p", "n": 1025, "m": 2048, "channels": 4, "dtype": "f32",
         "jitter": 0.25, "shape": "quadratic"},
        # projFEMq: steps of the loop with quadratic shape functions both ways
        {"name": "loop_f32", "kind": "loop", "n": 257, "m": 512, "channels": 1, "dtype": "f32",
         "solve": "refined", "jitter": 0.25, "shape": "quadratic", "m2p": "quadratic", "steps": 3},
        # fitting particle values and positions to a mesh field, the gradient configuration
        {"name": "grad_f32", "kind": "grad", "n": 1025, "m": 2048, "channels": 1, "dtype": "f32",
         "solve": "f32", "jitter": 0.25, "shape": "quadratic", "checkpoint": False, "back": False},
        # the gradient of a whole round trip in FP64 with checkpointed weights
        {"name": "grad_trip_f64", "kind": "grad", "n": 257, "m": 512, "channels": 2, "dtype": "f64",
         "solve": "f64", "jitter": 0.25, "shape": "quadratic", "checkpoint": True, "back": True},
        # many uneven problems at once
        {"name": "batch_f32", "kind": "batch", "count": 48, "n_lo": 65, "n_hi": 513, "sizes": 4,
         "channels": 3, "dtype": "f32", "solve": "refined", "jitter": 0.3, "shape": "quadratic"},
    ]


def trip(name, n, m, channels, dtype, solve, jitter=0.25, shape="quadratic", m2p="linear"):
    c = {"kind": "trip", "n": n, "m": m, "channels": channels, "dtype": dtype, "solve": solve,
         "jitter": jitter, "shape": shape, "m2p": m2p}
    return dict(c, name=name) if name else c


def draw(rng):
    """A case of the ranges above: mesh sizes over the logarithm, the configurations' particle densities
    (1, 2, sqrt(6) or 4 per spacing), every storage type, solve and shape function in use."""
    kind = rng.choice(["trip", "trip", "trip", "trip", "random", "m2p", "loop", "grad", "batch"])
    dtype = rng.choice(["f32", "f32", "f32", "f64", "bf16"])
    channels = rng.randint(1, 8) if rng.random() < 0.5 else rng.choice([1, 3, 4])
    density = rng.choice([1.0, 2.0, 2.0, math.sqrt(6.0), 4.0])
    jitter = rng.choice([0.25, 0.25, 0.3, round(rng.uniform(0.05, 0.3), 3)])

    def sizes(lo, hi, most):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n, max(40, min(most, int(round(density * (n - 1)))))

    if kind == "trip":
        solve = "f64" if dtype == "f64" else rng.choice(["refined", "refined", "refined", "f32", "refined_ff", "f64"])
        n, m = sizes(33, 769 if solve == "f64" else 2049, 1536 if solve == "f64" else 5000)
        return trip(None, n, m, channels, dtype, solve, jitter, rng.choice(["quadratic"] * 4 + ["linear"]),
                    "quadratic" if rng.random() < 0.25 else "linear")
    if kind == "random":
        n, m = sizes(129, 513, 1024)
        m = max(m, 256)
        return trip(None, n, m, channels, "f32", rng.choice(["refined", "refined", "f32"]), None,
                    rng.choice(["quadratic", "quadratic", "linear"]))
    if kind == "m2p":
        n, m = sizes(33, 2049, 4096)
        return {"kind": "m2p", "n": n, "m": m, "channels": channels, "dtype": dtype, "jitter": jitter,
                "shape": rng.choice(["linear", "quadratic"])}
    if kind == "loop":
        dtype = rng.choice(["f32", "f32", "f64"])
        n, m = sizes(33, 513, 1024)
        return {"kind": "loop", "n": n, "m": m, "channels": channels, "dtype": dtype,
                "solve": "f64" if dtype == "f64" else "refined", "jitter": min(jitter, 0.25),
                "shape": "quadratic", "m2p": rng.choice(["linear", "quadratic"]), "steps": rng.randint(1, 4)}
    if kind == "grad":
        dtype = rng.choice(["f32", "f32", "f64"])
        n, m = sizes(33, 1025 if dtype == "f32" else 385, 2048 if dtype == "f32" else 768)
        return {"kind": "grad", "n": n, "m": m, "channels": min(channels, 4), "dtype": dtype, "solve": dtype,
                "jitter": min(jitter, 0.25), "shape": rng.choice(["quadratic"] * 3 + ["linear"]),
                "checkpoint": rng.random() < 0.4, "back": rng.random() < 0.5}
    return {"kind": "batch", "count": rng.randint(3, 40), "n_lo": rng.randint(33, 65),
            "n_hi": rng.randint(97, 385), "sizes": rng.randrange(1000), "channels": min(channels, 4),
            "dtype": "f64" if dtype == "f64" else "f32", "solve": "f64" if dtype == "f64" else "refined",
            "jitter": jitter, "shape": "quadratic"}


def problem_sizes(case):
    """(n, particles per side) of each problem of a batch, or of the one problem."""
    if case["kind"] != "batch":
        return [(case["n"], case["m"])]
    r = random.Random(case["sizes"])
    got = []
    for _ in range(case["count"]):
        n = r.randint(case["n_lo"], case["n_hi"])
        got.append((n, (n - 1) * r.choice([1, 2, 4])))
    return got


# ---------------------------------------------------------------- inputs

def positions(m, jitter, dtype, gen):
    if jitter is None:
        return torch.rand(m * m, 2, dtype=torch.float64, device=DEVICE, generator=gen).to(dtype)
    u = torch.rand(m * m, 2, dtype=torch.float64, device=DEVICE, generator=gen)
    i = torch.arange(m * m, device=DEVICE)
    x = (torch.stack([i % m, i // m], 1) + 0.5 + jitter * (2 * u - 1)) / m
    return (x - x.floor()).to(dtype)


def fields(xy, channels, gen):
    """Taylor-Green velocity and pressure, a slotted disk and a density step, with a phase of the seed's."""
    x, y = xy[:, 0].double(), xy[:, 1].double()
    got = []
    for c in range(channels):
        a, b = (2 * math.pi * torch.rand(2, dtype=torch.float64, device=DEVICE, generator=gen)).unbind()
        k = 2 * math.pi * (1 + c // 4)
        if c % 4 == 0:
            f = torch.sin(k * x + a) * torch.cos(k * y + b)
        elif c % 4 == 1:
            f = -torch.cos(k * x + a) * torch.sin(k * y + b)
        elif c % 4 == 2:
            f = 0.25 * (torch.cos(2 * k * x + a) + torch.cos(2 * k * y + b))
        else:
            disk = ((x - 0.5) ** 2 + (y - 0.75) ** 2 <= 0.15 ** 2) & ~(((x - 0.5).abs() < 0.025) & (y < 0.85))
            f = disk.double() * (1 + 0.25 * torch.sin(a))
        got.append(f)
    return torch.stack(got, 1)


def mesh_nodes(n):
    g = torch.arange(n, dtype=torch.float64, device=DEVICE) % (n - 1) / (n - 1)
    return torch.stack([g.repeat(n), g.repeat_interleave(n)], 1)


def inputs(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    t = DTYPES[case["dtype"]]
    pos_t = torch.float64 if t == torch.float64 else torch.float32
    C = case["channels"]
    if case["kind"] == "batch":
        pos = [positions(m, case["jitter"], pos_t, gen) for _, m in problem_sizes(case)]
        return {"pos": torch.cat(pos), "vals": torch.cat([fields(p, C, gen).to(t) for p in pos])}
    n = case["n"]
    s = {"pos": positions(case["m"], case["jitter"], pos_t, gen)}
    if case["kind"] in ("m2p", "loop"):
        s["mesh"] = fields(mesh_nodes(n), C, gen).to(t).view(n, n, C)
    if case["kind"] == "loop":
        # a Taylor-Green velocity, half a cell a step
        vel = fields(mesh_nodes(n), 2, gen).to(pos_t).view(n, n, 2)
        s["vel"], s["dt"] = vel, 0.5 / (n - 1)
    if case["kind"] in ("trip", "grad"):
        s["vals"] = fields(s["pos"], C, gen).to(t)
    if case["kind"] == "grad":
        # the field to fit: another phase, and noise
        target = fields(mesh_nodes(n), C, gen)
        s["target"] = (target + 0.01 * torch.randn(target.shape, dtype=torch.float64, device=DEVICE, generator=gen)).to(t).view(n, n, C)
    return s


def prepare(case, seed):
    s = inputs(case, seed)
    s["case"] = case
    if case["kind"] == "batch":
        s["batch"] = P.Batch([(n, m * m) for n, m in problem_sizes(case)], case["channels"], DTYPES[case["dtype"]], DEVICE)
    elif case["kind"] != "grad":
        s["proj"] = P.Projector(case["n"], case["m"] ** 2, case["channels"], pos_dtype=s["pos"].dtype, device=DEVICE)
    else:
        s["vals"].requires_grad_(True)
        s["pos"].requires_grad_(True)
    return s


def run(state):
    c = state["case"]
    shape = SHAPES[c["shape"]]
    if c["kind"] == "trip":
        proj = state["proj"]
        proj.build(state["pos"])
        mesh = proj.p2m(state["vals"], shape=shape, solve=SOLVES[c["solve"]])
        return {"mesh": mesh, "back": proj.m2p(state["pos"], mesh, shape=SHAPES[c["m2p"]])}
    if c["kind"] == "m2p":
        return {"back": state["proj"].m2p(state["pos"], state["mesh"], shape=shape)}
    if c["kind"] == "loop":
        pos, mesh = P.projection_loop(state["proj"], state["pos"], state["mesh"], state["vel"], state["dt"], c["steps"],
                                      m2p_shape=SHAPES[c["m2p"]], p2m_shape=shape, solve=SOLVES[c["solve"]])
        return {"pos": pos, "mesh": mesh}
    if c["kind"] == "grad":
        vals, pos = state["vals"], state["pos"]
        mesh = PA.p2m(vals, pos, c["n"], shape=shape, solve=SOLVES[c["solve"]], checkpoint=c["checkpoint"])
        loss = 0.5 * (mesh - state["target"]).square().sum()
        if c["back"]:
            loss = loss + 0.5 * PA.m2p(mesh, pos, c["n"]).square().sum()
        gv, gp = torch.autograd.grad(loss, (vals, pos))
        return {"mesh": mesh.detach(), "grad_vals": gv, "grad_pos": gp}
    batch = state["batch"]
    back = batch.round_trip(state["pos"], state["vals"], shape=shape, solve=SOLVES[c["solve"]])
    return {"mesh": batch.mesh, "back": back}


def work(case):
    """Each input read once and each output written once; per node the three edge systems over about ten
    particles each (assembly, factor, solve, coefficients), per particle the six incircle tests of its star."""
    size = {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
    pos = 16 if case["dtype"] == "f64" else 8
    C, total, flops = case["channels"], 0, 0
    for n, m in problem_sizes(case):
        N, nodes = m * m, n * n
        p2m = 3 * (10 * 60 + 200) if case["shape"] == "quadratic" else 30
        if case["kind"] == "m2p":
            total += N * (pos + C * size) + nodes * C * size
            flops += N * (6 * C + (100 if case["shape"] == "quadratic" else 10))
            continue
        if case["kind"] == "loop":
            total += nodes * (2 * C * size + pos) + case["steps"] * N * 2 * pos
            flops += case["steps"] * (nodes * p2m + N * 6 * 30)
            continue
        grads = 2 if case["kind"] == "grad" else 0
        total += N * (pos * (1 + grads // 2) + C * size * (2 + grads // 2)) + nodes * C * size * (1 + grads // 2)
        flops += (1 + grads) * nodes * p2m + N * (6 * 30 + 6 * C)
    return {"bytes": total, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits, by plain torch
# Delaunay stars by gift wrapping over the nearest particles, the triangle of a node from the stars around it,
# and the coefficients of each edge by the normal equations with one step of refinement (ill-conditioned
# systems: the pseudo-inverse). Topology on coordinates rounded to 2^-32, as the framework defines it.

FULL = 1 << 32
STAR = 16


class Near:
    """The nearest particles of a point, from a grid of about two particles a cell."""

    def __init__(self, pos):
        self.q = torch.round(pos.double() * FULL).to(torch.int64) & (FULL - 1)
        self.N = self.q.shape[0]
        self.side = max(8, int(math.sqrt(self.N / 2)))
        cell = (self.q * self.side) >> 32
        cell = cell[:, 1] * self.side + cell[:, 0]
        count = torch.bincount(cell, minlength=self.side ** 2)
        order = torch.argsort(cell)
        rank = torch.arange(self.N, device=DEVICE) - (torch.cumsum(count, 0) - count)[cell[order]]
        self.table = torch.full((self.side ** 2, int(count.max())), -1, dtype=torch.int64, device=DEVICE)
        self.table[cell[order], rank] = order

    def offset(self, ids, at):
        d = (self.q[ids] - at) & (FULL - 1)
        return (d - (d >> 31) * FULL).double()

    def find(self, at, K, reach):
        """ids [B, K] by distance, their offsets, and the distance within which the list is complete."""
        c = (at * self.side) >> 32
        w = torch.arange(-reach, reach + 1, device=DEVICE)
        x, y = (c[:, :1] + w) % self.side, (c[:, 1:] + w) % self.side
        ids = self.table[(y[:, :, None] * self.side + x[:, None, :]).flatten(1)].flatten(1)
        d = self.offset(ids.clamp(min=0), at[:, None, :])
        l = torch.where(ids < 0, math.inf, d.square().sum(-1))
        l, k = torch.topk(l, min(K, l.shape[1]), dim=1, largest=False)
        clear = torch.minimum(l[:, -1].sqrt(), torch.tensor(reach * FULL / self.side, device=DEVICE, dtype=torch.float64))
        return torch.gather(ids, 1, k), torch.gather(d, 1, k[..., None].expand(-1, -1, 2)), clear

    def stars(self, who, K=40, reach=3):
        """Neighbours of each particle of `who`, counter-clockwise, -1 after the last; and whether proven."""
        ids, d, clear = self.find(self.q[who], K + 1, reach)
        ids, c = ids[:, 1:], d[:, 1:]                          # without itself
        valid = torch.isfinite(c[..., 0]) & (ids >= 0)
        rows = torch.arange(len(who), device=DEVICE)
        cur = torch.zeros(len(who), dtype=torch.int64, device=DEVICE)
        open_, ok, got = torch.ones_like(cur, dtype=torch.bool), torch.ones_like(cur, dtype=torch.bool), []
        for _ in range(STAR):
            got.append(torch.where(open_, ids[rows, cur], -1))
            w = c[rows, cur][:, None]
            cross = w[..., 0] * c[..., 1] - w[..., 1] * c[..., 0]
            cot = torch.where((cross > 0) & valid, ((c - w) * c).sum(-1) / cross, math.inf)
            best, nxt = cot.min(1)
            a, b = w[:, 0], c[rows, nxt]
            across = a.norm(dim=1) * b.norm(dim=1) * (a - b).norm(dim=1) / cross[rows, nxt]
            ok &= ~open_ | (torch.isfinite(best) & (across < clear))
            open_ = open_ & (nxt != 0)
            cur = nxt
        return torch.stack(got, 1), ok & ~open_

    def all_stars(self):
        got = []
        step = max(1024, (1 << 24) // (49 * self.table.shape[1]))
        for a in range(0, self.N, step):
            who = torch.arange(a, min(self.N, a + step), device=DEVICE)
            s, ok = self.stars(who)
            bad = (~ok).nonzero()[:, 0]
            for b in range(0, len(bad), 1024):                 # wide circles: far more neighbours
                part = bad[b:b + 1024]
                s[part], fine = self.stars(who[part], 400, min(14, self.side // 2 - 1))
                if not bool(fine.all()):
                    raise ValueError("a star could not be found")
            got.append(s)
        return torch.cat(got)

    def triangles(self, at, stars):
        """The Delaunay triangle that holds each point, counter-clockwise."""
        ids, _, _ = self.find(at, 24, 4)
        tri = torch.full((len(at), 3), -1, dtype=torch.int64, device=DEVICE)
        for k in range(ids.shape[1]):
            todo = (tri[:, 0] < 0).nonzero()[:, 0]
            if len(todo) == 0:
                return tri
            p = ids[todo, k]
            s = stars[p]
            nxt = torch.roll(s, -1, 1)
            nxt = torch.where(nxt < 0, s[:, :1], nxt)
            here = at[todo][:, None]
            o, a, b = self.offset(p[:, None], here), self.offset(s.clamp(min=0), here), self.offset(nxt.clamp(min=0), here)
            cr = lambda u, v: u[..., 0] * v[..., 1] - u[..., 1] * v[..., 0]  # noqa: E731
            inside = (cr(o, a) >= 0) & (cr(a, b) >= 0) & (cr(b, o) >= 0) & (s >= 0) & (p >= 0)[:, None]
            hit, j = inside.max(1)
            r = todo[hit]
            tri[r] = torch.stack([p[hit], s[hit, j[hit]], nxt[hit, j[hit]]], 1)
        raise ValueError("a node lies in no triangle")


def cholesky(M):
    """The function that solves M y = b (6 x 6, lists of tensors) by Cholesky, and the smallest pivot."""
    L = [[None] * 6 for _ in range(6)]
    least = None
    for j in range(6):
        s = M[j][j] - sum((L[j][k] ** 2 for k in range(j)), torch.zeros_like(M[j][j]))
        least = s.detach() if least is None else torch.minimum(least, s.detach())
        L[j][j] = s.clamp(min=1e-300).sqrt()
        for i in range(j + 1, 6):
            L[i][j] = (M[i][j] - sum((L[i][k] * L[j][k] for k in range(j)), torch.zeros_like(s))) / L[j][j]

    def back(v):
        z = []
        for r in range(6):
            z.append((v[r] - sum((L[r][k] * z[k] for k in range(r)), torch.zeros_like(v[r]))) / L[r][r])
        y = [None] * 6
        for r in reversed(range(6)):
            y[r] = (z[r] - sum((L[k][r] * y[k] for k in range(r + 1, 6)), torch.zeros_like(z[r]))) / L[r][r]
        return torch.stack(y, -1)

    return back, least


def monomials(x, y):
    return torch.stack([torch.ones_like(x), x, y, x * x, x * y, y * y], -1)


def edge_weights(d, ids, o):
    """A of the edge of the end offsets d[0], d[1], over the particles ids with offsets o (-1: none)."""
    valid = (ids >= 0).double()[..., None]
    mid, edge = 0.5 * (d[0] + d[1]), d[0] - d[1]
    s = edge.norm(dim=-1, keepdim=True)
    z = (o - mid[:, None]) / s[:, None]
    M6 = monomials(z[..., 0], z[..., 1]) * valid
    t = edge / s
    b = torch.stack([torch.zeros_like(t[:, 0])] * 3 + [-0.5 * t[:, 0] ** 2, -0.5 * t[:, 0] * t[:, 1], -0.5 * t[:, 1] ** 2], -1)
    G = M6.transpose(1, 2) @ M6
    solve, least = cholesky([[G[:, i, j] for j in range(6)] for i in range(6)])
    y = solve(list(b.unbind(-1)))
    y = y + solve(list((b - (M6.transpose(1, 2) @ (M6 @ y[..., None]))[..., 0]).unbind(-1)))
    A = (M6 @ y[..., None])[..., 0]
    poor = (least < 1e-6 * G.detach().diagonal(dim1=1, dim2=2).sum(-1)).nonzero()[:, 0]
    if len(poor):
        k = valid[poor, :, 0].sum(1).clamp(min=6)
        rows = torch.linalg.pinv(M6[poor].transpose(1, 2), rtol=k * 2.220446049250313e-16)
        A = A.clone()
        A[poor] = (rows @ b[poor][..., None])[..., 0]
    return A


class ExactP2M:
    """P2M onto the (n-1)^2 distinct nodes of a mesh, differentiable by values and positions."""

    def __init__(self, pos, n, shape):
        self.n, self.shape = n, shape
        self.near = Near(pos)
        self.stars = self.near.all_stars()
        nc = n - 1
        i = torch.arange(nc, device=DEVICE)
        fx = ((i << 32) + nc // 2) // nc
        self.at = torch.stack([fx.repeat(nc), fx.repeat_interleave(nc)], 1)
        self.xy = torch.stack([i.repeat(nc), i.repeat_interleave(nc)], 1).double() / nc

    def part(self, a, e, vals, pos):
        """Nodes a..e of the distinct ones, [e - a, C]."""
        with torch.no_grad():
            tri = self.near.triangles(self.at[a:e], self.stars)
        xy = self.xy[a:e]

        def off(ids):
            d = pos[ids] - xy[:, None]
            return d - d.detach().round()

        d = off(tri)
        cr = lambda u, v: u[..., 0] * v[..., 1] - u[..., 1] * v[..., 0]  # noqa: E731
        parts = torch.stack([cr(d[:, 1], d[:, 2]), cr(d[:, 2], d[:, 0]), cr(d[:, 0], d[:, 1])], 1)
        lam = parts / parts.sum(1, keepdim=True)
        out = (lam[..., None] * vals[tri]).sum(1)
        if self.shape == "linear":
            return out
        for k in range(3):
            f = (k + 1) % 3
            ids = torch.cat([self.stars[tri[:, k]], self.stars[tri[:, f]], tri[:, [k, f]]], 1).sort(1)[0]
            ids = torch.where(ids == torch.roll(ids, 1, 1), -1, ids)
            safe = ids.clamp(min=0)
            A = edge_weights((d[:, k], d[:, f]), ids, off(safe))
            out = out + 2 * (lam[:, k] * lam[:, f])[:, None] * (A[..., None] * vals[safe]).sum(1)
        return out

    def parts(self):
        nodes, step = len(self.at), 1 << 17
        return [(a, min(nodes, a + step)) for a in range(0, nodes, step)]

    def full(self, distinct):
        nc = self.n - 1
        m = distinct.view(nc, nc, -1)
        i = torch.arange(self.n, device=DEVICE) % nc
        return m[i][:, i]

    def __call__(self, vals, pos):
        return self.full(torch.cat([self.part(a, e, vals, pos) for a, e in self.parts()]))


def mesh_edge(ex, ey):
    """The ten nodes around the mesh edge from (0, 0) to (ex, ey) and their coefficients."""
    ring = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, -1)]
    nodes = sorted({(x, y) for x, y in ring} | {(x + ex, y + ey) for x, y in ring})
    s = math.hypot(ex, ey)
    z = (torch.tensor(nodes, dtype=torch.float64) - torch.tensor([ex, ey], dtype=torch.float64) / 2) / s
    tx, ty = ex / s, ey / s
    b = torch.tensor([0, 0, 0, -0.5 * tx * tx, -0.5 * tx * ty, -0.5 * ty * ty], dtype=torch.float64)
    return nodes, (torch.linalg.pinv(monomials(z[:, 0], z[:, 1]).T) @ b).tolist()


def exact_m2p(mesh, pos, shape):
    n = mesh.shape[0]
    nc = n - 1
    x = (pos - pos.detach().floor()) * nc
    i = x.detach().floor().clamp(max=nc - 1)
    s, t = (x - i).unbind(1)
    i, j = i.long().unbind(1)
    lower = s >= t
    # vertices (0,0), (1,0), (1,1) below the diagonal, (0,0), (1,1), (0,1) above it
    lam = torch.where(lower[:, None], torch.stack([1 - s, s - t, t], 1), torch.stack([1 - t, s, t - s], 1))
    at = lambda dx, dy, wrap: mesh[(j + dy) % nc if wrap else j + dy, (i + dx) % nc if wrap else i + dx]  # noqa: E731
    low = lower[:, None]
    out = lam[:, :1] * at(0, 0, False) + torch.where(low, lam[:, 1:2] * at(1, 0, False), lam[:, 2:] * at(0, 1, False)) \
        + torch.where(low, lam[:, 2:], lam[:, 1:2]) * at(1, 1, False)
    if shape == "linear":
        return out
    for is_low, edges in ((True, [((0, 0), (1, 0), 0, 1), ((1, 0), (1, 1), 1, 2), ((0, 0), (1, 1), 0, 2)]),
                          (False, [((0, 0), (1, 1), 0, 1), ((0, 1), (1, 1), 1, 2), ((0, 0), (0, 1), 0, 2)])):
        here = lower if is_low else ~lower
        for (ax, ay), (bx, by), u, v in edges:
            nodes, A = mesh_edge(bx - ax, by - ay)
            w = torch.where(here, 2 * lam[:, u] * lam[:, v], torch.zeros_like(s))[:, None]
            for (nx, ny), a in zip(nodes, A):
                out = out + a * w * at(ax + nx, ay + ny, True)
    return out


def exact_move(pos, vel, dt):
    half = pos + 0.5 * dt * exact_m2p(vel, pos, "linear")
    new = pos + dt * exact_m2p(vel, half, "linear")
    return new - new.floor()


def exact_grad(case, s):
    vals, pos = s["vals"].double().requires_grad_(True), s["pos"].double().requires_grad_(True)
    p = ExactP2M(s["pos"], case["n"], case["shape"])
    with torch.no_grad():
        mesh = p(vals, pos)
    gp = torch.zeros_like(pos)
    up = mesh - s["target"].double()
    if case["back"]:
        leaf = mesh.clone().requires_grad_(True)
        g = torch.autograd.grad(0.5 * exact_m2p(leaf, pos, "linear").square().sum(), (leaf, pos))
        up, gp = up + g[0], gp + g[1]
    # the image row and column are copies of the first ones
    up[0] += up[-1]
    up[:, 0] += up[:, -1]
    up = up[:-1, :-1].reshape(-1, up.shape[-1])
    gv = torch.zeros_like(vals)
    for a, e in p.parts():
        g = torch.autograd.grad((p.part(a, e, vals, pos) * up[a:e]).sum(), (vals, pos))
        gv, gp = gv + g[0], gp + g[1]
    return {"mesh": mesh, "grad_vals": gv, "grad_pos": gp}


def exact(case, seed):
    if sum(m * m for _, m in problem_sizes(case)) > 30_000_000:
        return None                                             # too long in 64 bits
    s = inputs(case, seed)
    if case["kind"] == "grad":
        return exact_grad(case, s)
    with torch.no_grad():
        if case["kind"] == "trip":
            pos = s["pos"].double()
            mesh = ExactP2M(s["pos"], case["n"], case["shape"])(s["vals"].double(), pos)
            return {"mesh": mesh, "back": exact_m2p(mesh, pos, case["m2p"])}
        if case["kind"] == "m2p":
            return {"back": exact_m2p(s["mesh"].double(), s["pos"].double(), case["shape"])}
        if case["kind"] == "loop":
            pos, mesh = s["pos"].double(), s["mesh"].double()
            for _ in range(case["steps"]):
                vals = exact_m2p(mesh, pos, case["m2p"])
                pos = exact_move(pos, s["vel"].double(), s["dt"])
                mesh = ExactP2M(pos, case["n"], case["shape"])(vals, pos)
            return {"pos": pos, "mesh": mesh}
        meshes, backs, at = [], [], 0
        for n, m in problem_sizes(case):
            pos, vals = s["pos"][at:at + m * m], s["vals"][at:at + m * m].double()
            mesh = ExactP2M(pos, n, case["shape"])(vals, pos.double())
            meshes.append(mesh.reshape(n * n, -1))
            backs.append(exact_m2p(mesh, pos.double(), "linear"))
            at += m * m
        return {"mesh": torch.cat(meshes), "back": torch.cat(backs)}
