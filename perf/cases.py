"""Performance cases: the work a program hands to this library, through its public entry points.

Every case is a dict of plain values.  ``op`` names the path, the other entries its sizes and options:

  csr        stored relation, sum or max reducer, forward or forward + backward (one training step of a layer)
  planned    stored relation whose feature table is far larger than L2, through its hot-source plan, with the
             degree histogram of the relation
  attention  online-softmax reducer over a stored relation
  radius     generated radius relation, Gaussian message (forward, or forward + backward) or the
             distance-weighted message (forward); the relation is rebuilt on every pass, as in a program whose
             points move
  lj         Lennard-Jones forces and energies, the relation rebuilt on every pass (one time step)
  mlp        edge network over a radius relation, forward + backward (one training step)
  knn        generated exact k-nearest-neighbour relation with a neighbour sum

Inputs are made on the GPU from the seed alone.  A program keeps its relation, its plan and its workspaces;
outputs are allocated by the calls.
"""
import math

import torch

from paper_2609_24802_b200 import api as T

DEV = "cuda"
CHUNK = 1 << 26          # edges handled at a time while a relation is generated


def listed():
    return [
        # a graph-learning layer on a skewed graph: sum aggregation with edge weights, forward + gradients
        {"name": "csr_sum_rmat", "op": "csr", "graph": "rmat", "n": 1 << 20, "degree": 16, "F": 64, "dtype": "f32",
         "weighted": True, "reducer": "sum", "backward": True, "index64": False},
        # the same layer with max aggregation
        {"name": "csr_max_rmat", "op": "csr", "graph": "rmat", "n": 1 << 20, "degree": 16, "F": 64, "dtype": "f32",
         "weighted": True, "reducer": "max", "backward": True, "index64": False},
        # a small simulation mesh inside a training loop: latency and launches count
        {"name": "csr_sum_mesh_small", "op": "csr", "graph": "mesh", "n": 16, "degree": 26, "F": 16, "dtype": "f32",
         "weighted": True, "reducer": "sum", "backward": True, "index64": False},
        # inference over a fixed-degree neighbour list, half-precision features, odd number of rows, a width that
        # does not fill a power of two of lanes
        {"name": "csr_sum_regular_f16", "op": "csr", "graph": "regular", "n": 131071, "degree": 32, "F": 40, "dtype": "f16",
         "weighted": False, "reducer": "sum", "backward": False, "index64": False},
        # the billion-edge relation held in device memory, 16-byte feature rows (the largest case)
        {"name": "csr_planned_billion", "op": "planned", "n": 1 << 26, "degree": 16, "F": 8, "dtype": "f16"},
        # graph attention on the skewed graph
        {"name": "attention_rmat", "op": "attention", "graph": "rmat", "n": 1 << 20, "degree": 16, "D": 64},
        # a few thousand points in a closed box (the smallest case): latency and launches count
        {"name": "radius_gauss_tiny", "op": "radius", "points": "uniform", "n": 4096, "F": 16, "message": "gauss",
         "neighbours": 3.6191, "periodic": False, "backward": True},
        # a million points in a periodic box, 32 neighbours each
        {"name": "radius_gauss_mid", "op": "radius", "points": "uniform", "n": 1000000, "F": 32, "message": "gauss",
         "neighbours": 32.0, "periodic": True, "backward": True},
        # distance-weighted sum of one scalar per point, rebuilt on every call
        {"name": "radius_dist_scalar", "op": "radius", "points": "uniform", "n": 131072, "F": 1, "message": "dist",
         "neighbours": 32.0, "periodic": False, "backward": False},
        # a molecular-dynamics force evaluation, four million particles
        {"name": "lj_lattice", "op": "lj", "m": 160, "jitter": 0.1},
        # an edge network trained on the vertices of a scanned surface
        {"name": "mlp_surface", "op": "mlp", "points": "surface", "n": 35947, "r": 0.015, "f_in": 8, "hidden": 32, "f_out": 4},
        # nearest-neighbour sum of one scalar per point
        {"name": "knn_scalar", "op": "knn", "points": "uniform", "n": 131072, "F": 1, "k": 16},
    ]


# ------------------------------------------------------------------------------ drawn cases
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _csr_sizes(rng, widths, most):
    """(rows, edges per row, width) with rows * edges * width at most `most`."""
    F = rng.choice(widths)
    degree = rng.choice((4, 8, 13, 16, 24, 32))
    return _log_int(rng, 500, max(1000, min(1 << 20, most // (degree * F)))), degree, F


def draw(rng):
    op = rng.choice(("csr", "csr", "csr", "csr", "planned", "attention", "radius", "radius", "radius", "lj", "mlp", "knn"))
    if op == "csr":
        dtype = rng.choice(("f32", "f32", "f16"))
        widths = (8, 12, 16, 24, 32, 48, 64, 100, 128) if dtype == "f32" else (8, 16, 24, 32, 40, 64, 128)
        n, degree, F = _csr_sizes(rng, widths, 1 << 30)
        graph = rng.choice(("rmat", "rmat", "regular", "mesh"))
        if graph == "mesh":
            n, degree = max(8, min(96, int(round((n * degree / 26.0) ** (1.0 / 3.0))))), 26
        return {"op": op, "graph": graph, "n": n, "degree": degree, "F": F, "dtype": dtype, "weighted": rng.random() < 0.7,
                "reducer": rng.choice(("sum", "sum", "max")), "backward": rng.random() < 0.6, "index64": rng.random() < 0.2}
    if op == "planned":
        dtype, F = rng.choice((("f16", 8), ("f16", 8), ("f16", 16), ("f32", 4), ("f32", 8)))
        return {"op": op, "n": _log_int(rng, 1 << 23, 1 << 25), "degree": rng.choice((8, 16)), "F": F, "dtype": dtype}
    if op == "attention":
        if rng.random() < 0.3:
            n = _log_int(rng, 64, 4096)
            return {"op": op, "graph": "causal", "n": n, "degree": n // 2 + 1, "D": rng.choice((32, 64, 128))}
        n, degree, D = _csr_sizes(rng, (16, 32, 48, 64, 100, 128), 1 << 30)
        return {"op": op, "graph": "rmat", "n": n, "degree": degree, "D": D}
    if op == "radius":
        message = rng.choice(("gauss", "gauss", "gauss", "dist"))
        points = rng.choice(("uniform", "uniform", "uniform", "surface", "clustered"))
        backward = message == "gauss" and rng.random() < 0.7
        F = rng.choice((4, 8, 16, 20, 32, 64)) if backward else rng.choice((1, 1, 3, 4, 8, 13, 16, 32, 64))
        if points == "clustered":
            return {"op": op, "points": points, "n": _log_int(rng, 1000, 40000), "F": min(F, 16), "message": message,
                    "neighbours": 2.0, "periodic": False, "backward": backward}
        neighbours = rng.choice((4.0, 8.0, 16.0, 32.0, 45.0))
        n = _log_int(rng, 1000, min(1000000, int((1 << 30) / (neighbours * max(F, 16)))))
        return {"op": op, "points": points, "n": n, "F": F, "message": message, "neighbours": neighbours,
                "periodic": points == "uniform" and rng.random() < 0.5, "backward": backward}
    if op == "lj":
        return {"op": op, "m": _log_int(rng, 8, 128), "jitter": round(rng.uniform(0.02, 0.1), 3)}
    if op == "mlp":
        n = _log_int(rng, 2000, 200000)
        return {"op": op, "points": "surface", "n": n, "r": round(0.015 * math.sqrt(35947.0 / n), 6), "f_in": rng.choice((1, 5, 8, 13)),
                "hidden": rng.choice((8, 16, 32)), "f_out": rng.choice((1, 3, 4))}
    points = rng.choice(("uniform", "uniform", "surface", "clustered"))
    return {"op": op, "points": points, "n": _log_int(rng, 1000, 100000 if points == "clustered" else 1000000),
            "F": rng.choice((1, 1, 3, 8, 16)), "k": rng.choice((4, 8, 16, 16, 32))}


# ------------------------------------------------------------------------------ inputs
def _bits(ids, p_one_if_0, p_one_if_1, levels, gen):
    """Ids whose bits are drawn one by one, each conditional on the same bit of `ids`."""
    out = torch.zeros_like(ids)
    for b in range(levels):
        u = torch.rand(ids.numel(), device=DEV, generator=gen)
        p = torch.where((ids >> b) & 1 == 1, p_one_if_1, p_one_if_0)
        out |= (u < p).to(ids.dtype) << b
    return out


def _rmat(n, n_edges, gen, index64=False):
    """Destination-oriented CSR of an R-MAT graph (a = 0.57, b = c = 0.19, d = 0.05), duplicates and self
    loops kept.  The bits of a row id are independent (one with probability c + d) and a column bit depends on
    the row bit of the same level only, so the degrees are drawn first and the columns row by row."""
    levels = max(1, (n - 1).bit_length())
    top = 1 << levels
    deg = torch.zeros(n + 1, dtype=torch.int64, device=DEV)

    def scaled(ids):
        return ids if n == top else (ids.long() * n >> levels).int()

    for e0 in range(0, n_edges, CHUNK):
        m = min(CHUNK, n_edges - e0)
        row = scaled(_bits(torch.zeros(m, dtype=torch.int32, device=DEV), 0.24, 0.24, levels, gen))
        deg[1:] += torch.bincount(row, minlength=n)
    rowptr = deg.cumsum(0)
    del deg
    col = torch.empty(n_edges, dtype=torch.int32, device=DEV)
    for e0 in range(0, n_edges, CHUNK):
        m = min(CHUNK, n_edges - e0)
        row = torch.searchsorted(rowptr, torch.arange(e0, e0 + m, device=DEV), right=True).int() - 1
        if n != top:
            row = ((row.long() << levels) // n).int()
        col[e0:e0 + m] = scaled(_bits(row, 0.25, 0.05 / 0.24, levels, gen))
    return rowptr if index64 else rowptr.int(), col


def _mesh(L, index64):
    """Hexahedral mesh of L^3 nodes: every node that shares an element, no self entries."""
    i = torch.arange(L, device=DEV)
    x, y, z = (t.reshape(-1, 1) for t in torch.meshgrid(i, i, i, indexing="ij"))
    o = torch.arange(27, device=DEV)
    o = o[o != 13]
    dx, dy, dz = o // 9 - 1, o // 3 % 3 - 1, o % 3 - 1
    X, Y, Z = x + dx, y + dy, z + dz
    ok = (X >= 0) & (X < L) & (Y >= 0) & (Y < L) & (Z >= 0) & (Z < L)
    rowptr = torch.zeros(L ** 3 + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = ok.sum(1).cumsum(0)
    return rowptr if index64 else rowptr.int(), ((X * L + Y) * L + Z)[ok].int()


def _relation(case, gen):
    n, degree, i64 = case["n"], case["degree"], case.get("index64", False)
    if case.get("graph") == "mesh":
        rowptr, col = _mesh(n, i64)
        n = n ** 3
    elif case.get("graph") == "causal":
        rowptr = torch.arange(n + 1, device=DEV)
        rowptr = (rowptr * (rowptr + 1) // 2).int()
        col = torch.tril_indices(n, n, device=DEV)[1].int()
    elif case.get("graph") == "regular":
        rowptr = torch.arange(n + 1, device=DEV) * degree
        rowptr = rowptr if i64 else rowptr.int()
        col = torch.randint(0, n, (n * degree,), device=DEV, dtype=torch.int32, generator=gen)
    else:
        rowptr, col = _rmat(n, n * degree, gen, i64)
    return T.CsrRelation(rowptr, col, n)


def _points(case, gen):
    n, kind = case["n"], case["points"]
    if kind == "uniform":
        return torch.rand((n, 3), device=DEV, generator=gen)
    if kind == "surface":          # a closed, bumpy surface inside the unit cube
        v = torch.randn((n, 3), device=DEV, dtype=torch.float64, generator=gen)
        v /= v.norm(dim=1, keepdim=True)
        rad = 0.34 + 0.05 * torch.sin(5.0 * v[:, 0]) * torch.cos(3.0 * v[:, 1]) + 0.04 * v[:, 2] ** 2
        return (0.5 + v * rad[:, None]).float()
    # most of the points in tight blobs, the rest a thin background
    nb, blobs = int(0.7 * n), 12
    centres = torch.rand((blobs, 3), device=DEV, generator=gen) * 0.8 + 0.1
    sigma = torch.rand(blobs, device=DEV, generator=gen) * 0.026 + 0.004
    which = torch.randint(0, blobs, (nb,), device=DEV, generator=gen)
    blob = centres[which] + torch.randn((nb, 3), device=DEV, generator=gen) * sigma[which, None]
    pos = torch.cat([blob, torch.rand((n - nb, 3), device=DEV, generator=gen)]).clamp_(0.0, 1.0 - 2.0 ** -24)
    return pos[torch.randperm(n, device=DEV, generator=gen)].contiguous()


def _randn(gen, *shape, dtype=torch.float32):
    return torch.randn(shape, device=DEV, generator=gen).to(dtype)


def _workspace(nbytes):
    return torch.empty(max(int(nbytes), 256), dtype=torch.uint8, device=DEV)


def _radius_of(case):
    """Cutoff with the stated mean number of neighbours (of a surface: on the surface)."""
    if case["points"] == "surface":
        return math.sqrt(case["neighbours"] * 1.6 / (math.pi * case["n"]))
    return (case["neighbours"] * 3.0 / (4.0 * math.pi * case["n"])) ** (1.0 / 3.0)


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    s = {"case": case, "op": case["op"]}
    if case["op"] in ("csr", "planned", "attention"):
        g = s["g"] = _relation(dict(case, index64=True) if case["op"] == "planned" else case, gen)
    if case["op"] == "csr":
        F, half = case["F"], case["dtype"] == "f16"
        s["reducer"] = T.SUM if case["reducer"] == "sum" else T.MAX
        s["x"] = _randn(gen, g.n_src, F, dtype=torch.float16 if half else torch.float32)
        # weights strictly inside (0, 1)
        s["w"] = torch.rand(g.n_edges, device=DEV, generator=gen).clamp_(min=2.0 ** -24) if case["weighted"] else None
        s["ws"] = _workspace(T.tiga_csr_workspace_bytes(g, F, T.F16 if half else T.F32, s["reducer"]))
        if case["backward"]:
            s["gy"] = _randn(gen, g.n_dst, F)
            s["ws_bwd"] = _workspace(T.tiga_csr_workspace_bytes(g, F, T.F16 if half else T.F32, s["reducer"], True))
    elif case["op"] == "planned":
        F, half = case["F"], case["dtype"] == "f16"
        s["x"] = _randn(gen, g.n_src, F, dtype=torch.float16 if half else torch.float32)
        s["plan"] = T.tiga_csr_plan_build(g, row_bytes=F * (2 if half else 4))
        s["ws"] = _workspace(T.tiga_csr_planned_workspace_bytes(s["plan"], F, T.F16 if half else T.F32, T.SUM))
    elif case["op"] == "attention":
        D = case["D"]
        s["q"], s["key"], s["value"] = (_randn(gen, g.n_dst, D) for _ in range(3))
        s["ws"] = _workspace(T.tiga_csr_attention_workspace_bytes(g, D))
    elif case["op"] == "radius":
        n, F = case["n"], case["F"]
        s["box"], s["periodic"], s["r"] = (1.0, 1.0, 1.0), (int(case["periodic"]),) * 3, _radius_of(case)
        s["pos"], s["x"] = _points(case, gen), _randn(gen, n, F)
        s["ws"] = _workspace(T.tiga_radius_workspace_bytes(n, F, s["r"], s["box"], s["periodic"], case["backward"]))
        if case["backward"]:
            s["gy"] = _randn(gen, n, F)
    elif case["op"] == "lj":
        m, a = case["m"], 0.8 ** (-1.0 / 3.0)
        L = torch.tensor(m * a, dtype=torch.float32).item()
        i = torch.arange(m, device=DEV, dtype=torch.float64) * a
        pos = torch.stack([t.reshape(-1) for t in torch.meshgrid(i, i, i, indexing="ij")], 1)
        pos += (torch.rand(pos.shape, device=DEV, dtype=torch.float64, generator=gen) * 2.0 - 1.0) * case["jitter"]
        pos = (pos - L * torch.floor(pos / L)).float()
        s["pos"] = torch.where(pos >= L, torch.zeros_like(pos), pos)
        s["box"], s["periodic"], s["r"] = (L, L, L), (1, 1, 1), 2.5
        s["ws"] = _workspace(T.tiga_radius_workspace_bytes(m ** 3, 4, s["r"], s["box"], s["periodic"]))
    elif case["op"] == "mlp":
        n, f_in, hidden, f_out = (case[k] for k in ("n", "f_in", "hidden", "f_out"))
        s["box"], s["periodic"], s["r"] = (1.0, 1.0, 1.0), (0, 0, 0), case["r"]
        s["pos"], s["x"], s["gy"] = _points(case, gen), _randn(gen, n, f_in), _randn(gen, n, f_out)

        def uniform(fan_in, *shape):
            return (torch.rand(shape, device=DEV, generator=gen) * 2.0 - 1.0) / math.sqrt(fan_in)

        s["net"] = (uniform(3 + f_in, hidden, 3 + f_in), uniform(3 + f_in, hidden), uniform(hidden, f_out, hidden), uniform(hidden, f_out))
        s["ws"] = _workspace(T.tiga_radius_workspace_bytes(n, f_in, s["r"], s["box"], s["periodic"], True))
    else:
        n = case["n"]
        s["box"], s["k"] = (1.0, 1.0, 1.0), case["k"]
        s["pos"], s["x"] = _points(case, gen), _randn(gen, n, case["F"])
        s["ws"] = _workspace(T.tiga_knn_workspace_bytes(n, s["k"], s["box"]))
    return s


# ------------------------------------------------------------------------------ one pass
def run(s):
    op, case = s["op"], s["case"]
    if op == "csr":
        out, arg = T.tiga_apply_csr(s["g"], s["x"], s["w"], s["reducer"], ws=s["ws"])
        if not case["backward"]:
            return out, arg
        gx, gw = T.tiga_apply_csr_backward(s["g"], s["x"], s["w"], s["gy"], s["reducer"], argmax=arg, want_w=case["weighted"], ws=s["ws_bwd"])
        return out, arg, gx, gw
    if op == "planned":
        out, _ = T.tiga_apply_csr_planned(s["plan"], s["x"], None, T.SUM, ws=s["ws"])
        return (out, *T.tiga_csr_degree_histogram(s["g"], 4096))
    if op == "attention":
        out, lse, _ = T.tiga_apply_csr_attention(s["g"], s["q"], s["key"], s["value"], case["D"] ** -0.5, ws=s["ws"])
        return out, lse
    if op == "radius":
        gauss, sigma = case["message"] == "gauss", 0.5 * s["r"]
        out, _, _ = T.tiga_apply_radius(s["pos"], s["x"], s["r"], s["box"], s["periodic"], T.MSG_GAUSS if gauss else T.MSG_DIST,
                                        p0=sigma, ws=s["ws"])
        if not case["backward"]:
            return out
        return (out, *T.tiga_apply_radius_backward(s["pos"], s["x"], s["gy"], s["r"], s["box"], s["periodic"], sigma, ws=s["ws"], reuse_plan=True))
    if op == "lj":
        return T.tiga_apply_radius(s["pos"], None, s["r"], s["box"], s["periodic"], T.MSG_LJ, p0=1.0, p1=1.0, ws=s["ws"])[0]
    if op == "mlp":
        out, _, _ = T.tiga_apply_radius_mlp(s["pos"], s["x"], s["r"], s["box"], s["periodic"], *s["net"], ws=s["ws"])
        return out, T.tiga_apply_radius_mlp_backward(s["pos"], s["x"], s["gy"], s["r"], s["box"], s["periodic"], *s["net"], ws=s["ws"], reuse_plan=True)
    return T.tiga_apply_knn(s["pos"], s["x"], s["k"], s["box"], ws=s["ws"])[:3]


# ------------------------------------------------------------------------------ work and tolerance
def work(case):
    """Every input read once, every output written once; the arithmetic of the messages and reductions."""
    op = case["op"]
    if op in ("csr", "planned", "attention"):
        n = case["n"] ** 3 if case.get("graph") == "mesh" else case["n"]
        E = n * case["degree"]
        if case.get("graph") == "mesh":
            E = (3 * case["n"] - 2) ** 3 - n
        elif case.get("graph") == "causal":
            E = n * (n + 1) // 2
        index = E * 4 + n * (8 if op == "planned" or case.get("index64") else 4)
        if op == "attention":
            D = case["D"]
            return {"bytes": index + 4 * n * (4 * D + 1), "flops": E * (4 * D + 4)}
        F, size, w = case["F"], 2 if case["dtype"] == "f16" else 4, 4 * E * case.get("weighted", False)
        b, f = index + w + n * F * (size + 4), E * F * (2 if w else 1)
        if op == "planned":
            return {"bytes": b, "flops": f}
        arg = 4 * n * F if case["reducer"] == "max" else 0
        b += arg
        if case["backward"]:
            b += index + 2 * w + n * F * (size + 4 + 4) + arg
            f += (E if case["reducer"] == "sum" else n) * F * (4 if w else 2)
        return {"bytes": b, "flops": f}
    if op == "lj":
        n = case["m"] ** 3
        return {"bytes": n * 28, "flops": n * 0.5 * 52.0 * 30}
    n = case["n"]
    if op == "radius":
        F, pairs = case["F"], n * case["neighbours"]
        b, f = n * (12 + 8 * F), pairs * (2 * F + 10)
        if case["backward"]:
            b += n * (24 + 12 * F)
            f += pairs * (6 * F + 16)
        return {"bytes": b, "flops": f}
    if op == "mlp":
        pairs = n * 15.0
        net = case["hidden"] * (3 + case["f_in"] + case["f_out"])
        return {"bytes": n * (48 + 12 * case["f_in"] + 8 * case["f_out"]), "flops": pairs * net * 8}
    return {"bytes": n * (12 + 8 * case["F"] + 8 * case["k"]), "flops": n * case["k"] * (case["F"] + 8.0)}


# About four times the distance of one pass from the same pass evaluated in fp64 (2-norm; largest entry).  The
# spread between the paths is the length of their sums: the hottest source of a skewed graph adds up tens of
# thousands of terms in an order of its own, a lattice particle's force is what is left of fifty larger ones.
_TOLERANCE = {
    "csr": {"rel": 1e-6, "max": 4e-4}, "csr_sum_backward": {"rel": 1e-5, "max": 5e-3}, "planned": {"rel": 1e-6, "max": 4e-4},
    "attention": {"rel": 1e-6, "max": 1e-5}, "radius": {"rel": 1e-6, "max": 1e-5}, "lj": {"rel": 6e-6, "max": 4e-5},
    "mlp": {"rel": 1e-5, "max": 4e-5}, "knn": {"rel": 5e-7, "max": 2e-6},
}


def tolerance(case):
    """Whole numbers (edge positions, neighbour ids, degree counts) and max results are the same."""
    if case["op"] == "csr" and case["reducer"] == "sum" and case["backward"]:
        return dict(_TOLERANCE["csr_sum_backward"])
    return dict(_TOLERANCE[case["op"]])
