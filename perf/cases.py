"""Timed cases of the library: one pass of each is what a user's program calls, through the Python binding.

A case is a dict of plain values:
  op      "knn"      kdt_knn / kdt_fcp on a tree that the program keeps (k = 1 goes through kdt_fcp)
          "ball"     kdt_radius_search (count, offsets, fill)
          "box"      kdt_box_search
          "density"  kdt_radius_reduce with a payload (photon-map density)
          "rebuild"  kdt_rebuild of a kept tree on moved points, then kdt_tree_export
          "build"    kdt_build of a new tree, kdt_tree_export, kdt_free
          "forest"   kdt_knn_batched over many small trees
  points  "uniform" in [0,1]^D, "clusters" (64 Gaussians of sigma 0.01), "surface" (256 spheres and tori)
  N, D, Q, k, r   points, dimensions, queries, neighbours, radius (0 in a knn case: unbounded)
  order   "none", "morton" or "cost" (KDT_MORTON | KDT_COST_ORDER)
  widest  the tree stores each node's split dimension (KDT_BUILD_WIDEST)
  T       number of trees of a forest case

Inputs are drawn on the GPU with the recipes of paper_2210_12859_gb300/synth.py.
"""
import math

import torch

from paper_2210_12859_gb300 import kdt

ORDER = {"none": 0, "morton": kdt.KDT_MORTON, "cost": kdt.KDT_MORTON | kdt.KDT_COST_ORDER}
PAYLOAD = 3  # RGB power of a photon


def case(name, op, points, N, D=3, Q=0, k=1, r=0.0, order="none", widest=False, T=1):
    c = {"op": op, "points": points, "N": N, "D": D, "Q": Q, "k": k, "r": r, "order": order, "widest": widest, "T": T}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one closest-point step of a scan registration: a small scan, no reordering, latency counts
        case("fcp_scan", "knn", "surface", 10007, Q=5003),
        # the small uniform workload: neighbourhoods of a 16 k point set
        case("knn_small", "knn", "uniform", 1 << 14, Q=1 << 14, k=8, order="morton"),
        # the paper's rig: uniform points in [0,1]^4, ten million closest points
        case("fcp_uniform4", "knn", "uniform", 1 << 22, D=4, Q=10_000_000, order="morton"),
        # neighbourhoods on scanned surfaces (normal estimation), an odd size
        case("knn_surface", "knn", "surface", 4_000_037, Q=4_000_037, k=16, order="morton"),
        # the benchmark workload: clustered points, a tenth of the queries between the clusters
        case("knn_clusters", "knn", "clusters", 1 << 24, Q=1 << 24, k=8, order="cost"),
        # large neighbourhoods in a bounded radius (density estimation)
        case("knn_k40_radius", "knn", "clusters", 1_500_001, Q=700_001, k=40, r=0.02, order="cost"),
        # feature vectors of eight dimensions
        case("knn_8d", "knn", "uniform", 200_003, D=8, Q=1 << 17, k=10, order="morton"),
        # fixed-radius neighbour lists (particle interactions)
        case("ball_search", "ball", "clusters", 1 << 22, Q=1_000_003, r=0.002, order="morton"),
        # photon map: density around the visible points of an image
        case("photon_density", "density", "surface", 300_007, Q=1 << 18, r=0.004, order="morton"),
        # points that move every frame: the tree of a kept size built anew
        case("rebuild_small", "rebuild", "uniform", 20_011),
        # a new tree of the largest set
        case("build_large", "build", "clusters", 1 << 24),
        # many uneven clouds, each with its own queries, in one call
        case("forest_clouds", "forest", "clusters", 4_000_000, Q=4_000_000, k=8, order="morton", T=300),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["knn", "knn", "knn", "knn", "ball", "box", "density", "rebuild", "build", "forest"])
    points = rng.choice(["uniform", "clusters", "surface"])
    order = rng.choice(["none", "morton", "cost"])
    widest = rng.random() < 0.2
    if op in ("build", "rebuild"):
        D = rng.choice([1, 2, 3, 3, 3, 4, 6, 8])
        if D != 3 and points == "surface":
            points = "uniform"
        return case("", op, points, _log_int(rng, 1_000, (1 << 23) * 3 // max(D, 3)), D=D, widest=widest and D <= 3)
    if op == "forest":
        T = _log_int(rng, 4, 400)
        n = _log_int(rng, 50 * T, max(4_000_000, 100 * T))
        return case("", op, "clusters", n, Q=n, k=rng.choice([1, 4, 8, 16, 24]), order=rng.choice(["none", "morton"]), T=T)
    if op != "knn":
        N = _log_int(rng, 5_000, 4_000_000)
        Q = _log_int(rng, 1_000, 1_000_000)
        # about `hits` points in a ball where the points are dense
        hits = math.exp(rng.uniform(math.log(2), math.log(100)))
        if points == "uniform":
            r = (hits / N / 4.19) ** (1 / 3)
        elif points == "clusters":
            r = 0.02 * (hits / N * 64) ** (1 / 3)
        else:
            r = 1.3 * (hits / N) ** 0.5
        return case("", op, points, N, Q=Q, r=round(r, 6), order=rng.choice(["none", "morton"]), widest=widest)
    D = rng.choice([2, 3, 3, 3, 3, 4, 6, 8])
    if D != 3 and points == "surface":
        points = "uniform"
    if D > 4:
        points = "uniform"
    most = {2: 1 << 23, 3: 1 << 23, 4: 1 << 22}.get(D, 200_000)
    N = _log_int(rng, 1_000, most)
    Q = _log_int(rng, 1_000, most)
    k = rng.choice([1, 1, 2, 5, 8, 8, 16, 20, 32])
    if points == "clusters" and (k > 16 or D == 4 or order == "none"):
        N, Q = min(N, 1 << 21), min(Q, 1 << 20)  # the queries between the clusters are long
    r = rng.choice([0.0, 0.0, 0.0, round(rng.uniform(0.005, 0.05), 4)])
    return case("", "knn", points, N, D=D, Q=Q, k=k, r=r, order=order if Q > 50_000 else rng.choice(["none", order]),
                widest=widest and D <= 3)


# ---- inputs


def _uniform(n, D, g):
    return torch.rand((n, D), generator=g, device="cuda")


def _clusters(n, D, g, centres, sigma):
    comp = torch.randint(0, centres.shape[0], (n,), generator=g, device="cuda")
    return centres[comp] + sigma * torch.randn((n, D), generator=g, device="cuda")


def _surface_shapes(g):
    S = 256
    u = torch.rand((S, 6), generator=g, device="cuda")
    R = 0.01 + 0.09 * u[:, 3]
    r = R * (0.2 + 0.3 * u[:, 4])
    torus = u[:, 5] < 0.5
    axis = torch.nn.functional.normalize(torch.randn((S, 3), generator=g, device="cuda"), dim=1)
    area = torch.where(torus, 4 * math.pi**2 * R * r, 4 * math.pi * R * R)
    return u[:, :3], R, r, torus, axis, area


def _surface(n, g, shapes):
    centre, R, r, torus, axis, area = shapes
    at = torch.cumsum(area.double(), 0)
    s = torch.searchsorted(at, torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * at[-1])
    s = s.clamp_(max=len(area) - 1)
    v = torch.nn.functional.normalize(torch.randn((n, 3), generator=g, device="cuda"), dim=1)
    a = axis[s]
    # torus: a point of the tube around the circle of radius R in the plane of `axis`
    flat = torch.nn.functional.normalize(v - (v * a).sum(1, keepdim=True) * a, dim=1)
    t = 2 * math.pi * torch.rand((n, 1), generator=g, device="cuda")
    tube = (R[s, None] + r[s, None] * torch.cos(t)) * flat + r[s, None] * torch.sin(t) * a
    p = centre[s] + torch.where(torus[s, None], tube, R[s, None] * v)
    return p + 1e-4 * torch.randn((n, 3), generator=g, device="cuda")


def _cloud_offsets(T, total, g):
    """T clouds of log-uniform sizes, 2^8 to 2^18 before they are scaled to `total` points."""
    w = torch.exp2(8 + 10 * torch.rand(T, generator=g, device="cuda", dtype=torch.float64))
    off = torch.round(torch.cumsum(w, 0) / w.sum() * total).to(torch.int64).cpu()
    return torch.cat([torch.zeros(1, dtype=torch.int64), off]).numpy()


def _data(c, seed):
    """(points, queries, second array or None)"""
    g = torch.Generator(device="cuda").manual_seed(seed * 7919 + 17)
    N, D, Q = c["N"], c["D"], c["Q"]
    if c["op"] == "forest":
        T = c["T"]
        off = _cloud_offsets(T, N, g)
        size = torch.from_numpy(off[1:] - off[:-1]).cuda()
        tree = torch.repeat_interleave(torch.arange(T, device="cuda"), size)
        centres = torch.rand((T, 8, D), generator=g, device="cuda")
        parts = torch.randint(1, 9, (T,), generator=g, device="cuda")
        sigma = 0.005 * 10 ** torch.rand((T, 8, 1), generator=g, device="cuda")
        both = []
        for _ in range(2):
            m = (torch.rand(N, generator=g, device="cuda") * parts[tree]).long()
            both.append(centres[tree, m] + sigma[tree, m] * torch.randn((N, D), generator=g, device="cuda"))
        return both[0], both[1], off
    if c["points"] == "uniform":
        p = _uniform(N, D, g)
        q = 1.2 * _uniform(Q, D, g) - 0.1 if N < 100_000 else _uniform(Q, D, g)
    elif c["points"] == "clusters":
        centres = torch.rand((64, D), generator=g, device="cuda")
        p = _clusters(N, D, g, centres, 0.01)
        q = _clusters(Q, D, g, centres, 0.01)
        far = torch.rand((Q, 1), generator=g, device="cuda") < 0.1
        q = torch.where(far, _uniform(Q, D, g), q)
    else:
        shapes = _surface_shapes(g)
        p, q = _surface(N, g, shapes), _surface(Q, g, shapes)
    extra = None
    if c["op"] == "box":
        extra = c["r"] * (0.5 + _uniform(Q, D, g))
    elif c["op"] == "density":
        extra = torch.rand((N, PAYLOAD), generator=g, device="cuda")
    return p.contiguous(), q.contiguous(), extra


def _hits(c):
    """About the hits of a pass: what balls of this radius hold where the points are dense."""
    N, r = c["N"], c["r"]
    if c["points"] == "uniform":
        hits = 4.19 * r**3 * N
    elif c["points"] == "clusters":
        hits = 0.75 * N / 64 * (r / 0.02) ** 3
    else:
        hits = N * (r / 1.3) ** 2
    return int(min(N, hits) * c["Q"])


def prepare(c, seed):
    p, q, extra = _data(c, seed)
    s = {"c": c, "q": q, "flags": ORDER[c["order"]], "r": c["r"] or math.inf}
    opts = kdt.KDT_BUILD_WIDEST if c["widest"] else 0
    if c["op"] == "forest":
        s["forest"] = kdt.kdt_build_batched(p, extra)
        s["off"] = extra
    elif c["op"] == "build":
        s["p"], s["opts"] = p, opts
    else:
        s["tree"] = kdt.kdt_build(p, opts)
        if c["op"] == "rebuild":
            s["p"] = p.flip(0).contiguous()
        elif c["op"] == "density":
            kdt.kdt_tree_set_payload(s["tree"], extra)
        elif c["op"] in ("ball", "box"):
            # the program's neighbour list: room for the hits of any step, filled to the front
            room = int(1.5 * _hits(c)) + 16 * c["Q"]
            s["ids"] = torch.zeros(room, dtype=torch.int32, device="cuda")
            if c["op"] == "ball":
                s["d2"] = torch.zeros(room, device="cuda")
            else:
                s["lo"], s["hi"] = q - extra, q + extra
    return s


def _keep(room, found):
    n = min(room.shape[0], found.shape[0])
    room[:n].copy_(found[:n])
    return room


def run(s):
    c = s["c"]
    op = c["op"]
    if op == "knn":
        if c["k"] == 1:
            return kdt.kdt_fcp(s["tree"], s["q"], s["r"], s["flags"])
        return kdt.kdt_knn(s["tree"], s["q"], c["k"], s["r"], s["flags"])
    if op == "ball":
        off, ids, d2 = kdt.kdt_radius_search(s["tree"], s["q"], c["r"], s["flags"])
        return off, _keep(s["ids"], ids), _keep(s["d2"], d2)
    if op == "box":
        off, ids = kdt.kdt_box_search(s["tree"], s["lo"], s["hi"], s["flags"])
        return off, _keep(s["ids"], ids)
    if op == "density":
        return kdt.kdt_radius_reduce(s["tree"], s["q"], c["r"], kdt.KDT_REDUCE_DENSITY, s["flags"], with_counts=True)
    if op == "rebuild":
        kdt.kdt_rebuild(s["tree"], s["p"])
        return kdt.kdt_tree_export(s["tree"])
    if op == "build":
        tree = kdt.kdt_build(s["p"], s["opts"])
        out = kdt.kdt_tree_export(tree)
        tree.free()
        return out
    return kdt.kdt_knn_batched(s["forest"], s["q"], s["off"], c["k"], s["r"], s["flags"])


def work(c):
    N, D, Q, k = c["N"], c["D"], c["Q"], c["k"]
    points = 4 * D * N
    if c["op"] in ("build", "rebuild"):
        # points in, coordinates and ids out; a comparison per point and level
        return {"bytes": 2 * points + 4 * N, "flops": N * max(1, int(math.log2(N)))}
    if c["op"] in ("knn", "forest"):
        # the tree (at most the neighbours that are reported, where these are fewer), the queries, the result rows
        return {"bytes": min(points + 4 * N, (4 * D + 4) * Q * k) + 4 * D * Q + 8 * k * Q, "flops": 3 * D * Q * k}
    hits = _hits(c)
    tree = min(points + 4 * N, (4 * D + 4) * hits)
    if c["op"] == "density":
        return {"bytes": tree + min(N, hits) * 4 * PAYLOAD + 4 * D * Q + (4 * PAYLOAD + 4) * Q, "flops": (3 * D + PAYLOAD) * hits}
    if c["op"] == "box":
        return {"bytes": tree + 8 * D * Q + 8 * Q + 4 * hits, "flops": 2 * D * hits}
    return {"bytes": tree + 4 * D * Q + 8 * Q + 8 * hits, "flops": 3 * D * hits}


# ---- the same in 64 bits, by comparing every query with every point


def exact(c, seed):
    if c["op"] not in ("knn", "density") or c["N"] * c["Q"] > 1 << 37:
        return None
    p, q, extra = _data(c, seed)
    P, Qs = p.double(), q.double()
    N, k = P.shape[0], c["k"]
    rows = max(1, (1 << 28) // N)
    # the radius that the call sees is a float32
    r2 = torch.tensor(c["r"] or math.inf, dtype=torch.float32).double().item() ** 2
    out = []
    for a in range(0, Qs.shape[0], rows):
        d2 = torch.zeros((min(rows, Qs.shape[0] - a), N), dtype=torch.float64, device="cuda")
        for j in range(P.shape[1]):
            d2 += (Qs[a:a + rows, j, None] - P[None, :, j]).square_()
        if c["op"] == "density":
            out.append((d2 <= r2).double() @ extra.double() / (math.pi * r2))
        else:
            v = torch.topk(d2, min(k, N), dim=1, largest=False, sorted=True).values
            v = torch.where(v <= r2, v, math.inf)
            out.append(torch.nn.functional.pad(v, (0, k - v.shape[1]), value=math.inf))
    res = torch.cat(out)
    if c["op"] == "density":
        return res, None
    return None, res[:, 0] if k == 1 else res
