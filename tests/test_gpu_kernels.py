"""Kernel variants and dispatch rules at the sizes where they could go wrong, against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from workloads import generators as G

pytestmark = pytest.mark.gpu

# FP32: the storage rounding of a value, at most 24 products and sums of a node and the rounding of
# their weights, each 2^-24 of the largest value times the weights' sum of magnitudes (below 1.3)
TOL32 = 2e-6
TOL64 = 1e-12


@pytest.fixture(scope="module")
def P():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1610_05266_gb300 as P
    return P


def relerr(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


def uniform(n, m, seed):
    pos = G.uniform01(G.SEED_BASE + seed, 2 * m * m).reshape(m * m, 2)
    return G.Problem("uniform", n, m, 0.0, 0, pos, G.taylor_green(pos))


PROBLEMS = {"tiny": lambda: G.config_tiny(), "odd": lambda: G.scaled_config("tg", 38, 91, 0.3),
            "coarse": lambda: G.scaled_config("tg", 41, 40, 0.3), "dense": lambda: G.scaled_config("tg", 33, 128),
            "uniform": lambda: uniform(65, 256, 900)}


@pytest.mark.parametrize("which", sorted(PROBLEMS))
def test_refined_solves(P, which):
    """Both refined solves form the residual in 64-bit fixed point: the same mesh bit for bit, within
    the FP32 bound of the oracle, on lattices of one to sixteen particles per node and on uniform
    random particles (long thin stencils, ill-conditioned systems)."""
    pr = PROBLEMS[which]()
    pos = torch.tensor(pr.pos, dtype=torch.float32, device="cuda")
    vals = torch.tensor(pr.vals, dtype=torch.float32, device="cuda")
    proj = P.Projector(pr.n, pr.N, C=pr.C, pos_dtype=torch.float32)
    proj.build(pos)
    a = proj.p2m(vals, solve=P.PFEM_SOLVE_F32_REFINED)
    b = proj.p2m(vals, solve=P.PFEM_SOLVE_F32_REFINED_FF)
    proj.check()
    assert torch.equal(a, b)
    ref = O.p2m(pr.n, pos.double().cpu().numpy(), vals.double().cpu().numpy(), shape=1, nthreads=8)
    assert relerr(a.cpu().numpy(), ref) <= TOL32


@pytest.mark.parametrize("C", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_mesh_quadratic_m2p(P, C, dtype):
    """Mesh QCSF M2P for every component count, on particles of both triangles of a cell, the first
    and last rows and columns among them, reading the distinct nodes only (the image row and
    column hold something else)."""
    n, N = 38, 4097
    pos = G.uniform01(G.SEED_BASE + 910, 2 * N).reshape(N, 2)
    pos[:64, 0] = np.repeat([0.0, 1e-7, 1.0 - 1e-7, 0.999], 16)
    pos[64:128, 1] = np.repeat([0.0, 1e-7, 1.0 - 1e-7, 0.999], 16)
    pos[128:160, 1] = pos[128:160, 0]
    pos = torch.tensor(pos, dtype=dtype, device="cuda")
    mesh = G.uniform01(G.SEED_BASE + 911, n * n * C).reshape(n, n, C)
    mesh[-1], mesh[:, -1] = mesh[0], mesh[:, 0]
    mesh = torch.tensor(mesh, dtype=dtype, device="cuda")
    proj = P.Projector(n, N, C=C, pos_dtype=dtype)
    spoilt = mesh.clone()
    spoilt[-1] = 7.0
    spoilt[:, -1] = 7.0
    got = proj.m2p(pos, spoilt, shape=P.PFEM_SHAPE_QUADRATIC)
    ref = O.m2p_quadratic(n, pos.double().cpu().numpy(), mesh.double().cpu().numpy())
    assert relerr(got.cpu().numpy(), ref) <= (TOL64 if dtype == torch.float64 else TOL32)


def _disk(M, R, fill, seed):
    """M x M lattice with the disk of radius R emptied and refilled with `fill` uniform particles."""
    pos = G.jittered_lattice(M, 0.2, G.SEED_BASE + seed)
    d = pos - 0.5
    d -= np.rint(d)
    pos = pos[(d ** 2).sum(1) >= R * R]
    u = G.uniform01(G.SEED_BASE + seed + 1, 2 * fill)
    r, a = R * np.sqrt(u[0::2]), 2 * np.pi * u[1::2]
    return np.concatenate([pos, 0.5 + np.stack([r * np.cos(a), r * np.sin(a)], 1)])


def _rays(M):
    """A lattice whose rows and columns are stretched unevenly: every particle shares its rays with
    others at different distances, at exactly equal angles."""
    g = np.cumsum(1.0 + 0.5 * (np.arange(M) % 3))
    g = np.floor((g - 0.5) / g[-1] * 4096) / 4096
    return np.stack([np.tile(g, M), np.repeat(g, M)], 1)


STARS = {"dense_disk": lambda: _disk(32, 0.1, 700, 920),      # lists over their capacity
         "sparse_disk": lambda: _disk(96, 0.06, 4, 930),      # circles wider than every list's cutoff
         "rays": lambda: _rays(33),                           # equal angles: the exact order
         "few": lambda: G.jittered_lattice(24, 0.3, G.SEED_BASE + 940),
         "ragged": lambda: G.jittered_lattice(37, 0.3, G.SEED_BASE + 941)[:-3]}


@pytest.mark.parametrize("which", sorted(STARS))
def test_stars_of_uneven_sets(P, which):
    """The list kernel and the warp search for queued stars, bit for bit against the oracle's stars."""
    pos = STARS[which]()
    proj = P.Projector(33, len(pos), pos_dtype=torch.float64)
    proj.build(torch.tensor(pos, device="cuda"))
    nbrs, counts = proj.stars()
    proj.check(which)
    nbrs, counts, perm = nbrs.cpu().numpy(), counts.cpu().numpy(), proj.cells.perm.cpu().numpy()
    cells = O.build_cells(33, pos)
    assert counts.sum() == 6 * len(pos)
    for s in range(len(pos)):
        mine, ref = list(perm[nbrs[s, :counts[s]]]), list(O.star(cells, int(perm[s])))
        assert mine[mine.index(min(mine)):] + mine[:mine.index(min(mine))] == \
            ref[ref.index(min(ref)):] + ref[:ref.index(min(ref))], s
        assert (nbrs[s, counts[s]:] == -1).all()


@pytest.mark.parametrize("which", sorted(PROBLEMS) + ["quad_end", "quad_past"])
def test_fp64_solves(P, which):
    """The FP32 factor with the solution refined in 64-bit fixed point: FP64 values within the FP64
    bound of the oracle and FP32 values within the FP32 bound, on both sides of the line between
    four lanes and one lane a node, with positions from other periods of the torus."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nodes = {"quad_end": 160 * sms, "quad_past": 160 * sms + 1}.get(which)
    if nodes:
        n = int(np.sqrt(nodes)) + (which == "quad_past")
        pr = G.scaled_config("tg", n, 2 * (n - 1))
    else:
        pr = PROBLEMS[which]()
    ref = O.p2m(pr.n, pr.pos, pr.vals, shape=1, nthreads=8)
    for shift in ((0.0, 0.0), (-3.0, 5.0)):
        pos = pr.pos + np.array(shift)
        want = ref if shift[0] == 0.0 else O.p2m(pr.n, pos, pr.vals, shape=1, nthreads=8)
        proj = P.Projector(pr.n, pr.N, C=pr.C, pos_dtype=torch.float64)
        proj.build(torch.tensor(pos, device="cuda"))
        mesh = proj.p2m(torch.tensor(pr.vals, device="cuda"))
        proj.check(which)
        assert relerr(mesh.cpu().numpy(), want) <= TOL64, shift
    pos = torch.tensor(pr.pos, dtype=torch.float32, device="cuda")
    proj = P.Projector(pr.n, pr.N, C=pr.C, pos_dtype=torch.float32)
    proj.build(pos)
    mesh = proj.p2m(torch.tensor(pr.vals, dtype=torch.float32, device="cuda"), solve=P.PFEM_SOLVE_F64)
    proj.check(which)
    assert relerr(mesh.cpu().numpy(), O.p2m(pr.n, pos.double().cpu().numpy(), pr.vals, shape=1, nthreads=8)) <= TOL32


@pytest.mark.parametrize("C", [1, 2, 3, 4, 7])
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
def test_linear_m2p_components_and_ends(P, C, dtype):
    """M2P for every component count and several particles a thread, with particles in the last cell, on
    cell boundaries and diagonals, from other periods, and a count that no block divides; a position
    that is not finite gives no finite value."""
    n, N = 38, 3001
    pos = G.uniform01(G.SEED_BASE + 950, 2 * N).reshape(N, 2)
    pos[:64, 0] = np.repeat([0.0, 1e-12, 1.0 - 1e-12, 36.0 / 37.0], 16)
    pos[64:128, 1] = np.repeat([0.0, 1e-12, 1.0 - 1e-12, 36.0 / 37.0], 16)
    pos[128:160, 1] = pos[128:160, 0]
    pos[200:300] += [-3.0, 5.0]
    pos_t = torch.float64 if dtype == "f64" else torch.float32
    pos = torch.tensor(pos, dtype=pos_t, device="cuda")
    mesh = G.uniform01(G.SEED_BASE + 951, n * n * C).reshape(n, n, C)
    mesh[-1], mesh[:, -1] = mesh[0], mesh[:, 0]
    mesh = torch.tensor(mesh, device="cuda").to({"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[dtype])
    proj = P.Projector(n, N, C=C, pos_dtype=pos_t)
    ref = O.m2p(n, pos.double().cpu().numpy(), mesh.double().cpu().numpy())
    # BF16: one rounding of the result, 2^-9; FP32 coordinates: 2^-24 n of a cell
    tol = {"f64": TOL64, "f32": n * 2.0 ** -23 + TOL32, "bf16": 2.0 ** -8}[dtype]
    assert relerr(proj.m2p(pos, mesh).double().cpu().numpy(), ref) <= tol
    pos[5, 0] = float("nan")
    assert not torch.isfinite(proj.m2p(pos, mesh)[5].float()).any()


def clustered(n, m, seed):
    """Half of the particles uniform, half in 64 normal clusters of standard deviation 0.02."""
    k = m * m // 2
    u = G.uniform01(G.SEED_BASE + seed, 2 * m * m + 2 * k + 128)
    a, r, c = u[:2 * (m * m - k)].reshape(-1, 2), u[2 * (m * m - k):-128][:2 * k].reshape(k, 2), u[-128:].reshape(64, 2)
    d = 0.02 * np.sqrt(-2 * np.log(1 - r[:, :1])) * np.stack([np.cos(2 * np.pi * r[:, 1]), np.sin(2 * np.pi * r[:, 1])], 1)
    p = c[np.arange(k) % 64] + d
    pos = np.concatenate([a, p - np.floor(p)])
    return G.Problem("clustered", n, m, 0.0, 0, pos, G.taylor_green(pos))


IRREGULAR = {"uniform": lambda: uniform(513, 1024, 71), "clustered": lambda: clustered(257, 512, 81)}


def noise(N, C=8):
    return 2.0 * G.uniform01(G.SEED_BASE + 960, C * N).reshape(N, C) - 1.0


def per_node(got, ref, w):
    """Largest error of a node over its weights' sum of magnitudes (values within one)."""
    n = ref.shape[0]
    return (np.abs(got - ref).max(-1) / np.abs(w).sum(-1).reshape(n, n)).max()


@pytest.mark.parametrize("which", sorted(IRREGULAR))
def test_fp64_weights_on_irregular_sets(P, which):
    """Explicit FP64 weights on particle sets with short edges beside wide stencils and ill-conditioned
    systems: at every node, not only where the mesh is largest, the image of white noise within
    FP64's 1e-12 of the oracle's, over the node's sum of weights."""
    pr = IRREGULAR[which]()
    v = noise(pr.N)
    proj = P.Projector(pr.n, pr.N, C=8, pos_dtype=torch.float64)
    proj.build(torch.tensor(pr.pos, device="cuda"))
    w_idx, w = proj.shape_weights()
    proj.check(which)
    got = proj.p2m(torch.tensor(v, device="cuda"), weights=(w_idx, w))
    ref = O.p2m(pr.n, pr.pos, v, shape=1, nthreads=16)
    assert per_node(got.cpu().numpy(), ref, w.cpu().numpy()) <= TOL64


@pytest.mark.parametrize("room", [0, 16])
def test_fp64_with_a_short_queue(P, room):
    """Uniform random particles, FP64, in a workspace whose fix-pass queue holds no or 16 nodes: about
    a hundred nodes' systems are beyond the FP32 factor, and the few that FP64's pivot
    tolerance queues still fit.  Without a queue exactly those report PFEM_ERR_DEGENERATE."""
    from paper_1610_05266_gb300 import api
    pr = uniform(129, 256, 970)
    proj = P.Projector(pr.n, pr.N, C=pr.C, pos_dtype=torch.float64)
    proj.build(torch.tensor(pr.pos, device="cuda"))
    c = proj.cells
    ws = torch.zeros(64 + room, dtype=torch.float64, device="cuda")
    mesh = torch.empty((pr.n, pr.n, pr.C), dtype=torch.float64, device="cuda")
    api.pfem_project_p2m(pr.n, proj.nb, pr.N, c.pos_sorted, c.q_sorted, c.cell_start, c.perm, pr.C,
                         torch.tensor(pr.vals, device="cuda"), P.PFEM_SHAPE_QUADRATIC, P.PFEM_SOLVE_F64,
                         None, None, 0, mesh, ws)
    code, detail = api.pfem_read_status(ws)
    mesh, ref = mesh.cpu().numpy(), O.p2m(pr.n, pr.pos, pr.vals, shape=1, nthreads=8)
    lost = ~np.isfinite(mesh).all(-1)
    if room:
        assert code == 0 and not lost.any(), (code, detail)
    else:
        assert lost.sum() <= 16 and (code == 5) == bool(lost.any())
    assert np.abs(mesh - ref)[~lost].max() <= TOL64 * np.abs(ref).max()


@pytest.mark.parametrize("route", ["p2m", "batch", "short_queue"])
@pytest.mark.parametrize("which", sorted(IRREGULAR))
def test_fp64_fix_pass_on_irregular_sets(P, which, route):
    """The nodes that the FP64 fast pass leaves to the fix pass (Cholesky with one refinement step, below
    its tolerance the SVD), in the table path, a batch and a call that searches the stars a node:
    the image of white noise at every node within FP64's 1e-12 of the oracle's over the node's sum of
    weights, which the unrefined normal equations of the worst of them miss a hundredfold."""
    from paper_1610_05266_gb300 import api
    pr = IRREGULAR[which]()
    v = noise(pr.N)
    pos, vals = torch.tensor(pr.pos, device="cuda"), torch.tensor(v, device="cuda")
    proj = P.Projector(pr.n, pr.N, C=8, pos_dtype=torch.float64)
    proj.build(pos)
    w = proj.shape_weights()[1]
    if route == "p2m":
        got = proj.p2m(vals)
        proj.check(which)
    elif route == "batch":
        b = P.Batch([(pr.n, pr.N)], 8, torch.float64, "cuda")
        b.build(pos)
        b.p2m(vals)
        got = b.mesh_view(0)
        assert b.status()[0] == 0
    else:
        c = proj.cells
        ws = torch.zeros(64 + pr.n * pr.n // 64, dtype=torch.float64, device="cuda")
        got = torch.empty((pr.n, pr.n, 8), dtype=torch.float64, device="cuda")
        api.pfem_project_p2m(pr.n, proj.nb, pr.N, c.pos_sorted, c.q_sorted, c.cell_start, c.perm, 8, vals,
                             P.PFEM_SHAPE_QUADRATIC, P.PFEM_SOLVE_F64, None, None, 0, got, ws)
        assert api.pfem_read_status(ws)[0] == 0
    ref = O.p2m(pr.n, pr.pos, v, shape=1, nthreads=16)
    assert per_node(got.cpu().numpy(), ref, w.cpu().numpy()) <= TOL64


def triangle_weights(pos, node, tri, stars):
    """Weights of a node in the triangle tri of particles with the given stars, by the pseudo-inverse."""
    d = pos - node

    def cr(a, b):
        return d[a][0] * d[b][1] - d[a][1] * d[b][0]

    lam = np.array([cr(tri[1], tri[2]), cr(tri[2], tri[0]), cr(tri[0], tri[1])])
    lam /= lam.sum()
    w = dict(zip(tri, lam))
    for e in range(3):
        f = (e + 1) % 3
        ids = sorted({tri[e], tri[f], *stars[e], *stars[f]})
        m, t = (d[tri[e]] + d[tri[f]]) / 2, d[tri[e]] - d[tri[f]]
        z, t = (d[ids] - m) / np.hypot(*t), t / np.hypot(*t)
        p = np.stack([np.ones(len(ids)), z[:, 0], z[:, 1], z[:, 0] ** 2, z[:, 0] * z[:, 1], z[:, 1] ** 2])
        A = np.linalg.pinv(p) @ np.array([0, 0, 0, -t[0] ** 2 / 2, -t[0] * t[1] / 2, -t[1] ** 2 / 2])
        for k, a in zip(ids, A):
            w[k] = w.get(k, 0.0) + 2 * lam[e] * lam[f] * a
    return w, lam


@pytest.mark.parametrize("seed", [26, 415, 1852])
def test_fp64_node_outside_a_sliver(P, seed):
    """A node among particles 1.6 units of 2^-32 apart: in the triangulation of the rounded positions it
    lies in a triangle that it is outside of, with coefficients 2 lambda lambda' of 4 to 16.  FP64 weights
    (of the triangle that was chosen) and P2M within 1e-12 of the largest."""
    n, I = 33, 8
    node = np.array([I, I]) / (n - 1)
    base = G.jittered_lattice(64, 0.2, G.SEED_BASE + 980)
    far = base[((base - node) ** 2).sum(1) > (1.2 / 64) ** 2]
    r = G.uniform01(G.SEED_BASE + 100000 + seed, 98).reshape(49, 2)
    g = np.stack(np.meshgrid(np.arange(7) - 3, np.arange(7) - 3), -1).reshape(49, 2)
    pos = np.concatenate([far, node + (1.6 * g + 0.7 * (2 * r - 1)) * 2.0 ** -32])
    proj = P.Projector(n, len(pos), C=1, pos_dtype=torch.float64)
    proj.build(torch.tensor(pos, device="cuda"))
    perm = proj.cells.perm.cpu().numpy()
    s, w = (x[I * n + I].cpu().numpy() for x in proj.shape_weights())
    got = dict(zip((int(k) for k in perm[s[s >= 0]]), w))
    tri = list(got)[:3]
    cells = O.build_cells(n, pos)
    ref, lam = triangle_weights(pos, node, tri, [[int(k) for k in O.star(cells, t)] for t in tri])
    assert max(abs(2 * lam[e] * lam[e - 1]) for e in range(3)) > 2 and set(got) == set(ref)
    top = max(abs(x) for x in ref.values())
    for k, x in ref.items():
        v = torch.zeros(len(pos), 1, dtype=torch.float64, device="cuda")
        v[k] = 1.0
        assert abs(got[k] - x) <= TOL64 * top and abs(proj.p2m(v)[I, I, 0].item() - x) <= TOL64 * top, (k, lam)


@pytest.mark.parametrize("d", [1e-4, 1e-9])
def test_fp64_weights_of_a_node_close_to_a_particle(P, d):
    """A node at distance d of a particle on 33^2 nodes: the other particles' weights, of the order of 32 d,
    within 1e-12 of the largest of them, by the table path's weights and P2M (four lanes a node), as FP64
    products give them (offsets from the node are exact here)."""
    n, (I, J) = 33, (16, 20)
    pos = G.jittered_lattice(64, 0.2, G.SEED_BASE + 990)
    node = np.array([I, J]) / 32
    close = int(((pos - node) ** 2).sum(1).argmin())
    pos[close] = node + d * np.array([1.0, 0.7])
    idx, ref = O.node_weights(O.build_cells(n, pos), I, J, 1)[:2]
    proj = P.Projector(n, len(pos), C=1, pos_dtype=torch.float64)
    proj.build(torch.tensor(pos, device="cuda"))
    perm = proj.cells.perm.cpu().numpy()
    s, w = (x[J * n + I].cpu().numpy() for x in proj.shape_weights())
    proj.check("weights")
    got = dict(zip((int(k) for k in perm[s[s >= 0]]), w))
    assert set(got) == {int(k) for k in idx}
    top = max(abs(x) for k, x in zip(idx, ref) if k != close)
    assert top < 100 * d
    for k, x in zip(idx, ref):
        v = torch.zeros(len(pos), 1, dtype=torch.float64, device="cuda")
        v[int(k)] = 1.0
        tol = TOL64 * (1.0 if k == close else top)
        assert abs(got[int(k)] - x) <= tol and abs(proj.p2m(v)[J, I, 0].item() - x) <= tol, int(k)
    proj.check("p2m")


def test_fp64_m2p_near_the_origin_of_a_fine_mesh(P):
    """FP64 particles in the first cell of 16385^2 nodes, where positions have bits below 2^-64: a linear field
    over that cell within 2^-52, three roundings of FP64 weights (the cell's side is a power of two, so the
    field's value is exact)."""
    n = 16385
    u = G.uniform01(G.SEED_BASE + 995, 2 * 4096).reshape(4096, 2)
    pos = u / (n - 1)
    mesh = torch.zeros(n, n, 1, dtype=torch.float64, device="cuda")
    mesh[:, 1:3] = 1.0
    got = torch.empty(len(pos), 1, dtype=torch.float64, device="cuda")
    from paper_1610_05266_gb300 import api
    api.pfem_interp_m2p(n, len(pos), torch.tensor(pos, device="cuda"), 1, mesh, got)
    assert np.abs(got[:, 0].cpu().numpy() - pos[:, 0] * (n - 1)).max() <= 2.0 ** -52


def test_linear_batches_of_two_block_shapes_in_two_threads(P):
    """Linear batched P2M with 64- and 256-thread blocks from two threads at once, each on its own stream: no
    launch is refused over shared memory that the other's shape does not need, and the meshes agree."""
    import threading
    pr = PROBLEMS["tiny"]()
    pos, vals = torch.tensor(pr.pos, device="cuda"), torch.tensor(pr.vals, device="cuda")
    got = {}

    def work(tile_rows):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                b = P.Batch([(pr.n, pr.N)] * 2, pr.C, torch.float64, "cuda")
                b.build(pos.repeat(2, 1))
                v = vals.repeat(2, 1)
                for _ in range(2000):
                    b.p2m(v, shape=P.PFEM_SHAPE_LINEAR, tile_rows=tile_rows)
                torch.cuda.current_stream().synchronize()
                assert b.status()[0] == 0
                got[tile_rows] = b.mesh.clone()
        except Exception as e:                   # reported by the main thread
            got[tile_rows] = e

    torch.cuda.synchronize()
    ts = [threading.Thread(target=work, args=(t,)) for t in (4, 16)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    for x in got.values():
        assert torch.is_tensor(x), x
    assert torch.equal(got[4], got[16])


@pytest.mark.parametrize("solve", ["F32", "F32_REFINED"])
def test_four_lanes_a_node_over_sets_of_both_sizes(P, solve):
    """Small meshes (four lanes a node) over uniform random particles, whose warps hold nodes with sets that fit
    shared memory next to larger ones: bit for bit what one lane a node gives that searches the stars
    itself, at the nodes which that solves without the fix pass (all but a few)."""
    from paper_1610_05266_gb300 import api
    pr, sv = uniform(97, 192, 996), getattr(P, "PFEM_SOLVE_" + solve)
    proj = P.Projector(pr.n, pr.N, C=pr.C, pos_dtype=torch.float32)
    proj.build(torch.tensor(pr.pos, dtype=torch.float32, device="cuda"))
    v = torch.tensor(pr.vals, dtype=torch.float32, device="cuda")
    four = proj.p2m(v, solve=sv)
    proj.check("table")
    c, one = proj.cells, torch.empty_like(four)
    api.pfem_project_p2m(pr.n, proj.nb, pr.N, c.pos_sorted, c.q_sorted, c.cell_start, c.perm, pr.C, v,
                         P.PFEM_SHAPE_QUADRATIC, sv, None, None, 0, one, torch.zeros(64, dtype=torch.float64, device="cuda"))
    done = torch.isfinite(one).all(-1)
    assert done.float().mean() > 0.97 and torch.equal(four[done], one[done])


@pytest.mark.parametrize("solve", ["F64", "F32", "F32_REFINED", "F32_REFINED_FF"])
def test_batch_totals_are_compared_for_every_solve(P, solve):
    """A node total other than the plan's: PFEM_ERR_INVALID_ARG with detail -1, the mesh untouched."""
    from paper_1610_05266_gb300 import api
    pr = PROBLEMS["tiny"]()
    pos, vals = (torch.tensor(x, dtype=torch.float32, device="cuda") for x in (pr.pos, pr.vals))
    b = P.Batch([(pr.n, pr.N)] * 2, pr.C, torch.float32, "cuda")
    b.build(pos.repeat(2, 1))
    b.mesh.fill_(7.0)
    api.pfem_batch_project_p2m(b.plan, b.nodes_total - 1, b.N_total, b.pos_sorted, b.q_sorted, b.cell_start, b.perm, pr.C,
                               vals.repeat(2, 1), P.PFEM_SHAPE_QUADRATIC, getattr(P, "PFEM_SOLVE_" + solve), b.mesh, 8,
                               64, b.ws)
    assert b.status() == (1, -1) and bool((b.mesh == 7.0).all())


LINEAR = {"uniform": lambda: uniform(70, 256, 901), "sparse": lambda: uniform(129, 60, 902),
          "dense_disk": lambda: G.Problem("disk", 37, 32, 0.0, 0, _disk(32, 0.1, 700, 920), None)}


@pytest.mark.parametrize("which", sorted(LINEAR))
def test_linear_on_irregular_sets(P, which):
    """Linear P2M, weights, adjoint and batches (all block shapes) where the hull leaves many stars to the
    warp, on meshes that leave lanes of a warp without a node, within FP64's bound of the oracle."""
    pr = LINEAR[which]()
    n, N, C = pr.n, len(pr.pos), 2
    v = noise(N, C)
    ref = O.p2m(n, pr.pos, v, shape=0, nthreads=8)
    pos, vals = torch.tensor(pr.pos, device="cuda"), torch.tensor(v, device="cuda")
    proj = P.Projector(n, N, C=C, pos_dtype=torch.float64)
    proj.build(pos)
    mesh = proj.p2m(vals, shape=P.PFEM_SHAPE_LINEAR)
    w = proj.shape_weights(shape=P.PFEM_SHAPE_LINEAR)
    proj.check(which)
    assert relerr(mesh.cpu().numpy(), ref) <= TOL64
    assert relerr(proj.p2m(vals, weights=w).cpu().numpy(), ref) <= TOL64
    g = 2.0 * G.uniform01(G.SEED_BASE + 961, n * n * C).reshape(n, n, C) - 1.0
    g[:, ::3] = 0.0                              # nodes without an upstream gradient
    gv, gp = proj.backward(vals, torch.tensor(g, device="cuda"), shape=P.PFEM_SHAPE_LINEAR)
    assert proj.backward_status()[0] == 0
    ov, op = O.p2m_backward(n, pr.pos, v, g, shape=0)
    assert relerr(gv.cpu().numpy(), ov) <= TOL64 and relerr(gp.cpu().numpy(), op) <= 1e-10
    b = P.Batch([(n, N)] * 2, C, torch.float64, "cuda")
    b.build(pos.repeat(2, 1))
    for rows in (4, 8, 16):
        b.mesh.fill_(float("nan"))
        b.p2m(vals.repeat(2, 1), shape=P.PFEM_SHAPE_LINEAR, tile_rows=rows)
        assert b.status()[0] == 0 and torch.equal(b.mesh_view(0), mesh) and torch.equal(b.mesh_view(1), mesh)


@pytest.mark.parametrize("M", [20, 37, 64])
def test_adjoint_of_few_particles_on_a_fine_mesh(P, M):
    """Particles with more entries than a thread sorts by itself (17 to several hundred): linear adjoint
    against the oracle, the same bits twice, and from checkpointed weights."""
    n = 65
    pos = G.jittered_lattice(M, 0.25, G.SEED_BASE + 997)
    N = len(pos)
    v, g = noise(N, 2), 2.0 * G.uniform01(G.SEED_BASE + 962, n * n * 2).reshape(n, n, 2) - 1.0
    proj = P.Projector(n, N, C=2, pos_dtype=torch.float64)
    proj.build(torch.tensor(pos, device="cuda"))
    vals, gm = torch.tensor(v, device="cuda"), torch.tensor(g, device="cuda")
    for shape in (0, 1):
        gv, gp = proj.backward(vals, gm, shape=shape)
        again = proj.backward(vals, gm, shape=shape)
        w = proj.shape_weights(shape=shape)
        cv, cp = proj.backward(vals, gm, shape=shape, weights=w)
        assert proj.backward_status()[0] == 0
        assert torch.equal(gv, again[0]) and torch.equal(gp, again[1]) and torch.equal(gp, cp)
        ov, op = O.p2m_backward(n, pos, v, g, shape=shape)
        assert relerr(gv.cpu().numpy(), ov) <= TOL64 and relerr(cv.cpu().numpy(), ov) <= TOL64
        assert relerr(gp.cpu().numpy(), op) <= TOL64
