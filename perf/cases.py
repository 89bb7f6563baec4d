"""What a user of the library has it do, as cases that can be timed.

Every case goes through the public calls of ``paper_2410_15227_gb300.api``.
The clouds are those of the library's own configurations: a sphere with
density ~ r^-1.5 times a lognormal turbulent field (sites drawn from the
particles), and the uniform cube.  A particle's smoothing length is
h = 1.2 n^(-1/3) with n the cloud's number density at its position, about 57
neighbours inside 2h.

Mixed precision (``precision=1``) computes weights in FP32 to 1e-5 relative:
its weights and what is summed from them are returned as the FP32 numbers a
program that asks for this mode keeps.  FP64 results are returned as FP64.
"""
import itertools
import math

import numpy as np
import torch

from paper_2410_15227_gb300 import api, inputs

H_FACT = 1.2
CUBE = (0.0, 1.0, 0.0, 1.0, 0.0, 1.0)
f64 = torch.float64


def listed():
    return [
        # the smallest ordinary call: 1,000 particles onto 1,000 cells in the
        # default FP64 mode, particles mapped directly; launches and host reads count
        dict(name="direct_cube_1k", kind="direct", n=1000, cells=1000),
        # many small snapshots at once, as a runtime study maps them
        dict(name="batch_16", kind="batch", snapshots=16, nmin=1000, nmax=20000),
        # the whole mapping step of one simulation output through
        # pseudo-particles, mixed precision: a fifth of the benchmark cloud,
        # the benchmark itself, and the largest configuration
        dict(name="step_200k", kind="step", n=200000, cells=52428, theta=0.12, sigma=1.0),
        dict(name="step_1m", kind="step", n=1000000, cells=262144, theta=0.065, sigma=1.0),
        dict(name="step_8m", kind="step", n=8000000, cells=2000000, theta=0.065, sigma=1.5),
        # the mapping alone on cells and pairs in hand (a new mass or h, the same
        # grid): particles directly in mixed precision, pseudo-particles in the
        # default FP64 mode
        dict(name="map_mixed_100k", kind="map", n=100000, cells=25000, theta=0.0, mixed=True),
        dict(name="map_fp64_200k", kind="map", n=200000, cells=52428, theta=0.12, mixed=False),
        # the grid on the benchmark's sites, read out for the radiative transfer
        dict(name="voronoi_262k", kind="voronoi", cells=262144, cloud="sphere"),
        # five Lloyd moves of a grid before the mapping; an odd number of sites
        dict(name="lloyd_30k", kind="lloyd", cells=30011, cloud="cube", iters=5),
        # gravity tree, adaptive walk and node smoothing lengths of the benchmark cloud
        dict(name="pseudo_1m", kind="pseudo", n=1000000, theta=0.065, h_tol=1e-13),
        # its particle-cell pairs
        dict(name="pairs_1m", kind="pairs", n=1000000, cells=262144, theta=0.065),
        # a cell field back onto pseudo-particles and particles (decode direction)
        dict(name="back_1m", kind="back", n=1000000, cells=262144, theta=0.065),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["direct", "batch", "step", "map", "voronoi", "lloyd", "pseudo", "pairs", "back"])
    if kind == "direct":
        return dict(kind=kind, n=_log(rng, 200, 20000), cells=_log(rng, 100, 20000))
    if kind == "batch":
        return dict(kind=kind, snapshots=rng.randint(2, 24), nmin=1000, nmax=_log(rng, 1500, 30000))
    if kind == "voronoi":
        return dict(kind=kind, cells=_log(rng, 500, 400000), cloud=rng.choice(["sphere", "cube"]))
    if kind == "lloyd":
        return dict(kind=kind, cells=_log(rng, 500, 100000), cloud=rng.choice(["sphere", "cube"]), iters=rng.randint(1, 5))
    n = _log(rng, 2000, 1000000 if kind != "map" else 200000)
    theta = round(0.065 * math.exp(rng.uniform(0.0, 1.5)), 4)
    if kind == "pseudo":
        return dict(kind=kind, n=n, theta=theta, h_tol=rng.choice([1e-13, 1e-13, 1e-2]))
    cells = max(64, int(n * rng.uniform(0.1, 0.3)))
    if kind == "step":
        return dict(kind=kind, n=n, cells=cells, theta=theta, sigma=rng.choice([1.0, 1.5]))
    if kind == "map":
        return dict(kind=kind, n=n, cells=cells, theta=rng.choice([0.0, max(theta, 0.1)]), mixed=rng.random() < 0.5)
    return dict(kind=kind, n=n, cells=cells, theta=theta)


# --- inputs -----------------------------------------------------------------

# A size has one cloud: the seed turns and mirrors it (one of the cube's 48
# symmetries) and puts particles and sites in another order, so that every
# seed is another input with as many nodes, faces and pairs.

def _gen(seed, k):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + k) % (1 << 62))
    return g


def _turned(p, seed, k):
    """p in another orientation and order, with the order taken."""
    rng = np.random.default_rng([int(seed), 7])
    axes, flip = rng.permutation(3).tolist(), rng.integers(0, 2, 3).tolist()
    order = torch.randperm(p.shape[0], generator=_gen(seed, k), device="cuda")
    p = p[order]
    return torch.stack([-p[:, a] if f else p[:, a] for a, f in zip(axes, flip)], 1), order


def _sphere(n, sigma):
    """(positions, smoothing lengths) of the n particles of the sphere cloud."""
    grf = torch.as_tensor(inputs.grf(2 if sigma == 1.0 else 5), device="cuda")
    gen, gmax, side = _gen(n, 1), grf.max(), grf.shape[0]
    out, dens, have, tried, factor = [], [], 0, 0, 0.0
    while have < n:
        b = int(min(max(8 * (n - have), 4096), 1 << 24))
        r = torch.rand(b, generator=gen, dtype=f64, device="cuda") ** (2.0 / 3.0)
        v = torch.randn(b, 3, generator=gen, dtype=f64, device="cuda")
        p = v * (r / v.norm(dim=1))[:, None]
        i = ((p + 1.0) * (0.5 * side)).long().clamp_(0, side - 1)
        g = grf[i[:, 0], i[:, 1], i[:, 2]]
        boost = torch.exp(sigma * (g - gmax))
        factor, tried = factor + float(boost.sum()), tried + b
        acc = torch.rand(b, generator=gen, dtype=f64, device="cuda") < boost
        out.append(p[acc])
        dens.append(1.5 / (4.0 * math.pi) * r[acc] ** -1.5 * boost[acc])
        have += out[-1].shape[0]
    p, d = torch.cat(out)[:n], torch.cat(dens)[:n] * (n * tried / factor)
    return p, H_FACT * d ** (-1.0 / 3.0)


def _cube(n, seed, k):
    p = torch.rand(n, 3, generator=_gen(n, k), dtype=f64, device="cuda")
    return _turned(p - 0.5, seed, k)[0] + 0.5


def _axes(p):
    return [p[:, k].contiguous() for k in range(3)]


def _sphere_box(p, h):
    L = float((p.abs().amax(dim=1) + 2.0 * h).max())
    return (-L, L, -L, L, -L, L)


def _sph_problem(n, cells, sigma, seed):
    p, h = _sphere(n, sigma)
    box = _sphere_box(p, h)
    sites = torch.randperm(n, generator=_gen(n, 2), device="cuda")[:cells]
    G, _ = _turned(p[sites], seed, 2)
    X, order = _turned(p, seed, 1)
    return dict(X=_axes(X), h=h[order], m=torch.full((n,), 1.0 / n, dtype=f64, device="cuda"), G=_axes(G), box=box,
                src=[(0.0, 0.0, 0.0)], f_cell=torch.rand(cells, generator=_gen(seed, 3), dtype=f64, device="cuda"))


def _params(case, mixed):
    theta = case.get("theta", 0.1)
    return api.Params(r_part=0.05, r_leaf=0.1, theta=theta if theta > 0 else 0.1, h_fact=H_FACT,
                      h_tol=case.get("h_tol", 1e-13), precision=1 if mixed else 0, fp64_threshold=1e-5)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind, ctx=api.Context(0))
    ctx = s["ctx"]
    if kind == "direct":
        n, cells = case["n"], case["cells"]
        s.update(X=_axes(_cube(n, seed, 4)), G=_axes(_cube(cells, seed, 5)), box=CUBE,
                 h=torch.full((n,), H_FACT * n ** (-1.0 / 3.0), dtype=f64, device="cuda"),
                 m=torch.full((n,), 1.0 / n, dtype=f64, device="cuda"),
                 f_cell=torch.rand(cells, generator=_gen(seed, 3), dtype=f64, device="cuda"), P=_params(case, False))
        return s
    if kind == "batch":
        rng = np.random.default_rng([case["snapshots"], case["nmax"], 6])
        snaps = []
        for k in range(case["snapshots"]):
            n = int(round(math.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"])))))
            q = _sph_problem(n, max(n // 4, 8), 1.0, int(seed) * 64 + k)
            snaps.append(dict(x=q["X"][0], y=q["X"][1], z=q["X"][2], m=q["m"], h=q["h"], gx=q["G"][0], gy=q["G"][1],
                              gz=q["G"][2], box=q["box"], sources=q["src"], f_cell=q["f_cell"]))
        s.update(snaps=snaps, P=_params(case, True))
        return s
    if kind in ("voronoi", "lloyd"):
        if case["cloud"] == "cube":
            s.update(G=_axes(_cube(case["cells"], seed, 5)), box=CUBE)
        else:
            p, h = _sphere(case["cells"], 1.0)
            s.update(G=_axes(_turned(p, seed, 5)[0]), box=_sphere_box(p, h))
        s.update(P=_params(case, True), iters=case.get("iters", 0))
        return s
    if kind == "pseudo":
        s.update(_sph_problem(case["n"], 8, 1.0, seed), P=_params(case, True))
        return s
    s.update(_sph_problem(case["n"], case["cells"], case.get("sigma", 1.0), seed))
    s["P"] = _params(case, case.get("mixed", True))
    if kind == "step":
        return s
    # cells (and pairs) in hand: pairs, map, back
    s["vor"] = api.build_voronoi(ctx, *s["G"], s["box"], s["P"])
    if case["theta"] > 0:
        s["tree"] = api.build_tree(ctx, *s["X"], s["m"], s["box"], 8)
        s["ps"] = api.make_pseudo_particles(ctx, s["tree"], s["h"], s["src"], s["P"])
        q = s["ps"].get()
        s["Q"] = [q["x"], q["y"], q["z"], q["h"], q["m"]]
    else:
        s["Q"] = [*s["X"], s["h"], s["m"]]
    if kind == "pairs":
        return s
    s["pr"] = api.find_pairs(ctx, *s["Q"][:4], s["vor"])
    if kind == "back":
        # weights of the pairs: the kernel at the site times the cell volume
        pr, v = s["pr"].get(), s["vor"].get()["volume"]
        i, j = pr["pair_i"].long(), pr["pair_j"].long()
        d2 = sum((s["Q"][k][i] - s["G"][k][j]) ** 2 for k in range(3))
        q = (d2.sqrt() / s["Q"][3][i]).clamp_(max=1.99)
        s["w"] = torch.where(q < 1, 1 - 1.5 * q * q + 0.75 * q ** 3, 0.25 * (2 - q) ** 3) * v[j] / (
            math.pi * s["Q"][3][i] ** 3)
    return s


# --- one pass ---------------------------------------------------------------

def run(s):
    ctx, P, kind = s["ctx"], s["P"], s["kind"]
    if kind == "batch":
        res, _ = api.map_batch(0, s["snaps"], P, nworkers=4)
        s["held"] = res   # read by the casts below: kept until the next pass
        return [dict(rho=r["rho"].float(), f=r["f"].float(), npseudo=r["npseudo"], npairs=r["npairs"]) for r in res]
    if kind == "voronoi":
        return api.build_voronoi(ctx, *s["G"], s["box"], P).get()
    if kind == "lloyd":
        return list(api.lloyd(ctx, *[g.clone() for g in s["G"]], s["box"], s["iters"], P))
    if kind == "pseudo":
        tree = api.build_tree(ctx, *s["X"], s["m"], s["box"], 8)
        ps = api.make_pseudo_particles(ctx, tree, s["h"], s["src"], P)
        return dict(tree=tree.get(), pseudo=ps.get())
    if kind == "pairs":
        return api.find_pairs(ctx, *s["Q"][:4], s["vor"]).get()
    if kind == "map":
        w, rho, wsum, _ = api.map_exact(ctx, s["pr"], *s["Q"], s["vor"], P, want_count=False)
        return [t.float() for t in (w, rho, wsum)] if P.precision else [w, rho, wsum]
    if kind == "back":
        f, fp = api.map_back(ctx, s["pr"], s["w"], s["f_cell"], s.get("ps"), s.get("tree"))
        num, den = api.map_back_sums(ctx, s["pr"], s["w"], s["f_cell"], torch.zeros_like(f), torch.zeros_like(f))
        return dict(f=f, particles=fp, num=num, den=den)
    if kind == "direct":
        vor = api.build_voronoi(ctx, *s["G"], s["box"], P)
        pr = api.find_pairs(ctx, *s["X"], s["h"], vor)
        w, rho, wsum, _ = api.map_exact(ctx, pr, *s["X"], s["h"], s["m"], vor, P, want_count=False)
        f, _ = api.map_back(ctx, pr, w, s["f_cell"])
        return dict(w=w, rho=rho, wsum=wsum, f=f)
    tree = api.build_tree(ctx, *s["X"], s["m"], s["box"], 8)
    ps = api.make_pseudo_particles(ctx, tree, s["h"], s["src"], P)
    vor = api.build_voronoi(ctx, *s["G"], s["box"], P)
    q = ps.get()
    pr = api.find_pairs(ctx, q["x"], q["y"], q["z"], q["h"], vor)
    w, rho, wsum, _ = api.map_exact(ctx, pr, q["x"], q["y"], q["z"], q["h"], q["m"], vor, P, want_count=False)
    f, fp = api.map_back(ctx, pr, w, s["f_cell"], ps, tree)
    return dict(w=w.float(), rho=rho.float(), wsum=wsum.float(), f=f.float(), particles=fp.float())


# --- work -------------------------------------------------------------------

# Per cell of a random site set: faces, and face-vertices.
FACES, FACE_VERTS = 15.5, 81.0
# Flops per pair of the closed form with every vertex, edge and face quantity
# formed once: 81 face-edges of about 100, and 16 faces of about 100.
PAIR_FLOPS = 10000.0
PAIRS_PER_CELL = 92.0      # pseudo-particles of the benchmark cloud, at 1e6 particles
PAIRS_PER_PARTICLE = 43.0  # particles mapped directly, a quarter as many cells


def work(case):
    """Inputs read once, outputs written once; the arithmetic of the closed form."""
    kind = case["kind"]
    n, c = case.get("n", 0), case.get("cells", 0)
    vor_bytes, vor_flops = c * (24 + 32 + FACES * 40 + FACE_VERTS * 24), c * 33.0 * 30 * 7
    tree_bytes, tree_flops = n * 40 * 1.5 + n * 0.41 * 88, n * 12 * 9.0 + 0.1 * n * 60 * 3 * 20.0
    if kind in ("direct", "map", "pairs", "back", "step"):
        if case.get("theta", 0.0) > 0:
            pairs = c * PAIRS_PER_CELL * (0.065 / case["theta"]) ** (0.0 if kind == "step" else 0.3)
        else:
            pairs = n * PAIRS_PER_PARTICLE * max(1.0, 4.0 * c / n) ** 0.7
    if kind == "batch":
        n = case["snapshots"] * (case["nmax"] - case["nmin"]) / math.log(case["nmax"] / case["nmin"])
        return dict(bytes=n * 48 + n / 4 * 40, flops=30 * n * PAIR_FLOPS)
    if kind == "voronoi":
        return dict(bytes=vor_bytes, flops=vor_flops)
    if kind == "lloyd":
        return dict(bytes=c * 48.0, flops=case["iters"] * vor_flops)
    if kind == "pseudo":
        return dict(bytes=tree_bytes, flops=tree_flops)
    if kind == "pairs":
        return dict(bytes=c * (FACES * 32 + FACE_VERTS * 24) + pairs * 9, flops=pairs * 200.0)
    if kind == "map":
        return dict(bytes=c * (FACES * 32 + FACE_VERTS * 24) + pairs * 16, flops=pairs * PAIR_FLOPS)
    if kind == "back":
        return dict(bytes=pairs * 16 + n * 12 + c * 8, flops=pairs * 6.0)
    if kind == "direct":
        return dict(bytes=n * 56 + c * 40 + pairs * 8, flops=pairs * PAIR_FLOPS + vor_flops)
    return dict(bytes=n * 56 + c * 40 + pairs * 4, flops=pairs * PAIR_FLOPS + vor_flops + tree_flops)


# --- the same numbers in plain torch, 64 bits --------------------------------

def _basis(A, B2, D, t):
    """Antiderivatives over tau of D A Q^k / (A^2 + tau^2) that the kernel's
    pieces need, at tau = t: (D atan, atan(D t / (A Q)), k = 2, 3, 4, 5)."""
    Q2 = B2 + t * t
    Q, B, D2 = Q2.sqrt(), B2.sqrt(), D * D
    ash, j0, psi = torch.asinh(t / B), torch.atan2(t, A), torch.atan2(D * t, A * Q)
    u1 = 0.5 * (t * Q + B2 * ash)
    j1 = A * ash + D * psi
    j3 = A * u1 + D2 * j1
    j2 = A * t + D2 * j0
    j4 = A * (A * A * t + t ** 3 / 3) + 2 * D2 * A * t + D2 * D2 * j0
    j5 = A * (0.25 * t * Q * Q2 + 0.75 * B2 * u1) + D2 * j3
    return D * j0, psi, D * j2, D * j3, D * j4, D * j5


def _phi(A, D, u, kD):
    """int_0^u [K(Q) - K(D)] D A / (A^2 + tau^2) dtau, Q^2 = D^2 + A^2 + tau^2."""
    B2 = D * D + A * A
    t1, t2 = (1 - B2).clamp(min=0).sqrt(), (4 - B2).clamp(min=0).sqrt()
    c1 = (0, 0, 1 / 6, 0, -3 / 40, 1 / 40)
    c2 = (-1 / 20, 1 / 60, 1 / 3, -1 / 4, 3 / 40, -1 / 120)
    c3 = (7 / 20, -1 / 4, 0, 0, 0, 0)
    total = -kD * D * torch.atan2(u, A)
    for c, hi, lo in ((c1, torch.minimum(u, t1), None), (c2, torch.minimum(torch.maximum(u, t1), t2), t1),
                      (c3, torch.maximum(u, t2), t2)):
        for sign, t in ((1, hi),) if lo is None else ((1, hi), (-1, lo)):
            for ck, bk in zip(c, _basis(A, B2, D, t)):
                if ck:
                    total = total + (sign * ck) * bk
    return total


def _K(q):
    k1 = q ** 2 / 6 - 3 * q ** 4 / 40 + q ** 5 / 40
    k2 = q ** 2 / 3 - q ** 3 / 4 + 3 * q ** 4 / 40 - q ** 5 / 120 + 1 / (60 * q.clamp(min=1)) - 1 / 20
    return torch.where(q < 1, k1, torch.where(q < 2, k2, 7 / 20 - 1 / (4 * q.clamp(min=1))))


def _weights(pi, pj, X, h, cell_off, nrm, dst, mnr, v0, v1):
    """w_ij of the pairs by the signed sum over the cells' face-edges [cell_off[j],
    cell_off[j+1]): face normal nrm and offset dst, in-plane outward edge normal
    mnr, end points v0, v1."""
    w = torch.zeros(pi.numel(), dtype=f64, device="cuda")
    cnt = cell_off[1:] - cell_off[:-1]
    step = max(1, (1 << 23) // max(1, int(cnt.double().mean())))
    for a in range(0, pi.numel(), step):
        i, j = pi[a:a + step], pj[a:a + step]
        c = cnt[j]
        who = torch.repeat_interleave(torch.arange(i.numel(), device="cuda"), c)
        e = torch.arange(who.numel(), device="cuda") - (c.cumsum(0) - c)[who] + cell_off[j][who]
        p, ih = X[i][who], 1 / h[i][who]
        sd = dst[e] - (nrm[e] * p).sum(1)
        sa = (mnr[e] * (v0[e] - p)).sum(1)
        ln = (v1[e] - v0[e]).norm(dim=1)
        ed = (v1[e] - v0[e]) / ln.clamp(min=1e-300)[:, None]
        T0 = (ed * (v0[e] - p)).sum(1) * ih
        T1 = T0 + ln * ih
        D, A = (sd.abs() * ih).clamp(min=1e-150), (sa.abs() * ih).clamp(min=1e-150)
        kD = _K(D)
        t = torch.sign(T1) * _phi(A, D, T1.abs(), kD) - torch.sign(T0) * _phi(A, D, T0.abs(), kD)
        w[a:a + step] = torch.zeros(i.numel(), dtype=f64, device="cuda").index_add_(
            0, who, torch.sign(sd) * torch.sign(sa) * t) / math.pi
    return w


def _edges_of(v, centres):
    """Face-edges of cells given by vertex loops (counter-clockwise faces)."""
    fvo, cfo = v["face_vert_off"], v["cell_face_off"]
    k = torch.arange(v["verts"].shape[0], device="cuda")
    face = torch.searchsorted(fvo, k, right=True) - 1
    nxt = torch.where(k + 1 < fvo[face + 1], k + 1, fvo[face])
    v0, v1, n = v["verts"], v["verts"][nxt], v["normals"][face]
    m = torch.linalg.cross(v1 - v0, n)
    m = m / m.norm(dim=1).clamp(min=1e-300)[:, None]
    return fvo[cfo], n, (n * v0).sum(1), m, v0, v1


def _cube_cells(G):
    """(offsets, face-edges, volumes) of the Voronoi cells of G in the unit
    cube from every triple of the walls and the nearest bisectors; None where
    those do not bound a cell."""
    nc, near = G.shape[0], min(96, G.shape[0] - 1)
    idx = torch.cdist(G, G).topk(near + 1, largest=False).indices[:, 1:]
    tri = torch.tensor(list(itertools.combinations(range(near + 6), 3)), device="cuda")
    wall = torch.tensor([[s if a == k else 0.0 for k in range(3)] for a in range(3) for s in (-1.0, 1.0)],
                        dtype=f64, device="cuda")
    parts = []
    for a in range(0, nc, 16):
        g = G[a:a + 16]
        r = G[idx[a:a + 16]] - g[:, None]
        ln = r.norm(dim=2)
        n = torch.cat([r / ln[..., None], wall.expand(g.shape[0], 6, 3)], 1)
        d = torch.cat([0.5 * ln, torch.stack([g[:, 0], 1 - g[:, 0], g[:, 1], 1 - g[:, 1], g[:, 2], 1 - g[:, 2]], 1)], 1)
        A, B, C = (n[:, tri[:, k]] for k in range(3))
        dA, dB, dC = (d[:, tri[:, k]][..., None] for k in range(3))
        bc, ca, ab = torch.linalg.cross(B, C), torch.linalg.cross(C, A), torch.linalg.cross(A, B)
        v = (dA * bc + dB * ca + dC * ab) / (A * bc).sum(2, keepdim=True)
        ok = torch.isfinite(v).all(2)
        for k in range(near + 6):
            ok &= (v * n[:, k, None]).sum(2) <= d[:, k, None] + 1e-12
        c, t = ok.nonzero(as_tuple=True)
        parts.append((c + a, tri[t], v[c, t] + g[c], n, d + (n * g[:, None]).sum(2)))
    cell, planes, vert = (torch.cat([p[k] for p in parts]) for k in range(3))
    n, d = (torch.cat([p[k] for p in parts]) for k in (3, 4))
    own = (vert - G[cell]).norm(dim=1)
    if bool((torch.cdist(vert, G).amin(dim=1) < own - 1e-9).any()):
        return None
    m = near + 6
    key = torch.cat([(cell * m + planes[:, x]) * m + planes[:, y] for x, y in ((0, 1), (0, 2), (1, 2))])
    vid = torch.arange(vert.shape[0], device="cuda").repeat(3)
    key, order = key.sort(stable=True)
    vid = vid[order]
    if key.numel() % 2 or bool((key[0::2] != key[1::2]).any()):
        return None
    key, v0, v1 = key[0::2], vert[vid[0::2]], vert[vid[1::2]]
    cell, x, y = key // (m * m), key // m % m, key % m
    cell, f, o = torch.cat([cell, cell]), torch.cat([x, y]), torch.cat([y, x])
    v0, v1 = torch.cat([v0, v0]), torch.cat([v1, v1])
    cell, order = cell.sort(stable=True)
    f, o, v0, v1 = f[order], o[order], v0[order], v1[order]
    nf, no, df = n[cell, f], n[cell, o], d[cell, f]
    mm = no - (no * nf).sum(1, keepdim=True) * nf
    mm = mm / mm.norm(dim=1, keepdim=True)
    off = torch.searchsorted(cell, torch.arange(nc + 1, device="cuda"))
    g = G[cell]
    vol = torch.zeros(nc, dtype=f64, device="cuda").index_add_(
        0, cell, (df - (nf * g).sum(1)) * _fan(g, nf, df, mm, v0, v1) / 3)
    return (off, nf, df, mm, v0, v1), vol


def _fan(g, nf, df, mm, v0, v1):
    """Signed area of the triangle (foot of g in the face, v0, v1)."""
    foot = g + (df - (nf * g).sum(1))[:, None] * nf
    return 0.5 * (mm * (v0 - foot)).sum(1) * (v1 - v0).norm(dim=1)


def exact(case, seed):
    kind = case["kind"]
    # grids of more than a few thousand sites, and what is mapped onto them,
    # would take minutes by exhaustive clipping
    if kind == "direct" and case["cells"] <= 2000 and case["n"] <= 4000:
        s = prepare(case, seed)
        X, G, h = torch.stack(s["X"], 1), torch.stack(s["G"], 1), s["h"]
        cells = _cube_cells(G)
        if cells is None:
            return None
        edges, vol = cells
        i, j = ((torch.cdist(X, G) < 0.75 + 2 * h[:, None]).nonzero(as_tuple=True))
        w = _weights(i, j, X, h, *edges)
        add = lambda at, k, v: torch.zeros(k, dtype=f64, device="cuda").index_add_(0, at, v)  # noqa: E731
        u = add(i, X.shape[0], w)
        return dict(w=None, rho=add(j, G.shape[0], s["m"][i] * w) / vol, wsum=u,
                    f=add(i, X.shape[0], w * s["f_cell"][j]) / u)
    if kind == "map":
        # cells and pairs are this case's inputs; the weights are computed here
        s = prepare(case, seed)
        v, pr = s["vor"].get(), s["pr"].get()
        i, j = pr["pair_i"].long(), pr["pair_j"].long()
        X, h, m = torch.stack(s["Q"][:3], 1), s["Q"][3], s["Q"][4]
        w = _weights(i, j, X, h, *_edges_of(v, s["G"]))
        rho = torch.zeros(case["cells"], dtype=f64, device="cuda").index_add_(0, j, m[i] * w) / v["volume"]
        return [w, rho, torch.zeros_like(h).index_add_(0, i, w)]
    if kind == "back":
        s = prepare(case, seed)
        pr = s["pr"].get()
        i, j = pr["pair_i"].long(), pr["pair_j"].long()
        num = torch.zeros_like(s["Q"][0]).index_add_(0, i, s["w"] * s["f_cell"][j])
        den = torch.zeros_like(num).index_add_(0, i, s["w"])
        q = s["ps"].get()
        f = num / den
        where = torch.zeros(case["n"], dtype=torch.long, device="cuda")
        where[q["first"].long()] = 1
        fp = torch.empty(case["n"], dtype=f64, device="cuda")
        fp[s["tree"].get()["perm"].long()] = f[where.cumsum(0) - 1]
        return dict(f=f, particles=fp, num=num, den=den)
    if kind == "pseudo":
        return _pseudo(case, seed)
    return None


def _pseudo(case, seed):
    """The tree-walk level by level and the node smoothing lengths with every
    neighbour sum over the whole population, plain torch."""
    s = prepare(case, seed)
    X, n, P = torch.stack(s["X"], 1), case["n"], s["P"]
    lo = torch.tensor(s["box"][0::2], dtype=f64, device="cuda")
    hi = torch.tensor(s["box"][1::2], dtype=f64, device="cuda")
    q = ((X - lo) * (2097152.0 / (hi - lo))).floor().clamp_(0, 2097151).long()
    key = torch.zeros(n, dtype=torch.long, device="cuda")
    for b in range(21):
        for k in range(3):
            key |= ((q[:, k] >> b) & 1) << (3 * b + 2 - k)
    key, perm = key.sort(stable=True)
    Xs, ms = X[perm], s["m"][perm]
    group, act = torch.zeros(n, dtype=torch.long, device="cuda"), torch.arange(n, device="cuda")
    first, emit = [], dict(first=[], x=[], m=[], h0=[], ext=[])
    pop_at, pop_x = [], []
    for level in range(22):
        if act.numel() == 0:
            break
        ng = int(group[-1]) + 1
        cnt = torch.bincount(group, minlength=ng)
        first = act[(cnt.cumsum(0) - cnt)]
        mass = torch.zeros(ng, dtype=f64, device="cuda").index_add_(0, group, ms[act])
        com = torch.zeros(ng, 3, dtype=f64, device="cuda").index_add_(0, group, ms[act, None] * Xs[act]) / mass[:, None]
        size = torch.zeros(ng, dtype=f64, device="cuda").scatter_reduce_(0, group, (Xs[act] - com[group]).norm(dim=1), "amax")
        r = com.norm(dim=1)
        leaf = (cnt <= 8) | (level == 21)
        ext = leaf & (r < P.r_part)
        opened = ~leaf & ((r < P.r_leaf) | (size > P.theta * r))
        node = ~ext & ~opened
        at = node[group].nonzero(as_tuple=True)[0]
        h0 = torch.where(cnt == 1, s["h"][perm[first]], 2 * P.h_fact * size)
        emit["first"].append(first[node]); emit["x"].append(com[node]); emit["m"].append(mass[node])
        emit["h0"].append(h0[node]); emit["ext"].append(torch.zeros(int(node.sum()), dtype=torch.bool, device="cuda"))
        at = act[ext[group]]
        emit["first"].append(at); emit["x"].append(Xs[at]); emit["m"].append(ms[at])
        emit["h0"].append(s["h"][perm[at]]); emit["ext"].append(torch.ones(at.numel(), dtype=torch.bool, device="cuda"))
        pop_at.append(first[~opened]); pop_x.append(com[~opened])
        keep = opened[group]
        act, group = act[keep], group[keep]
        if act.numel():
            digit = key[act] >> (3 * (20 - level)) if level < 21 else key[act]
            group = torch.cat([torch.zeros(1, dtype=torch.long, device="cuda"), (digit[1:] != digit[:-1]).long()]).cumsum(0)
    f = torch.cat(emit["first"])
    order = f.argsort()
    x, m, h0, ext = (torch.cat(emit[k])[order] for k in ("x", "m", "h0", "ext"))
    pop = torch.cat(pop_x)

    def sums(xa, ha):
        """S = sum of w(q) over the population, and h dS/dh."""
        S, dS = torch.empty_like(ha), torch.empty_like(ha)
        step = max(1, (1 << 27) // pop.shape[0])
        for a in range(0, ha.numel(), step):
            d = torch.zeros(xa[a:a + step].shape[0], pop.shape[0], dtype=f64, device="cuda")
            for k in range(3):
                d += (xa[a:a + step, k, None] - pop[None, :, k]) ** 2
            near = (d < 4 * ha[a:a + step, None] ** 2).nonzero(as_tuple=True)
            q = d[near].sqrt() / ha[a:a + step][near[0]]
            w = torch.where(q < 1, 1 - 1.5 * q ** 2 + 0.75 * q ** 3, 0.25 * (2 - q) ** 3)
            dw = torch.where(q < 1, 3 * q ** 2 - 2.25 * q ** 3, 0.75 * q * (2 - q) ** 2)
            zero = torch.zeros(d.shape[0], dtype=f64, device="cuda")
            S[a:a + step] = zero.index_add(0, near[0], w)
            dS[a:a + step] = zero.index_add(0, near[0], dw)
        return S, dS

    # Eq. 8 with n = S / (pi h^3) is S(h) = pi h_fact^3, S increasing in h
    h = h0.clone()
    todo = (~ext).nonzero(as_tuple=True)[0]
    if P.h_tol > 1e-10 or todo.numel() * pop.shape[0] > 12_000_000_000:
        h = None   # a loose tolerance's h is a point of the iteration, not the root
    else:
        lo_, hi_ = torch.zeros_like(h), torch.full_like(h, math.inf)
        for _ in range(60):
            S, dS = sums(x[todo], h[todo])
            ht, target = h[todo], math.pi * P.h_fact ** 3
            hi_[todo] = torch.where(S > target, torch.minimum(hi_[todo], ht), hi_[todo])
            lo_[todo] = torch.where(S < target, torch.maximum(lo_[todo], ht), lo_[todo])
            new = ht * torch.exp((target - S) / dS.clamp(min=1e-300)).clamp(0.5, 2.0)
            out = ~((new > lo_[todo]) & (new < hi_[todo]))
            mid = torch.where(hi_[todo] < math.inf, 0.5 * (lo_[todo] + hi_[todo]), 2 * ht)
            new = torch.where(out & (S != target), mid, new)
            h[todo] = new
            todo = todo[((new - ht).abs() > 1e-13 * ht) & (new != ht)]
            if todo.numel() == 0:
                break
    out = dict(x=x[:, 0], y=x[:, 1], z=x[:, 2], m=m, h=h)
    return dict(pseudo=out)
