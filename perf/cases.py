"""The colorings that stand for this library's use, one call through the public
entry points each: single distance-1, distance-2 and partial distance-2 calls on
device-resident graphs from the smallest to the largest the repository is
configured for, the batched call, and the server with a queue of requests.

Every input is made on the GPU by torch from the seed alone, by the recipes of
``paper_2107_00075_gb300.inputs`` (meshes, 2D grids, Erdos-Renyi, R-MAT, random
bipartite patterns).  The coloring seed of a call is the input seed, so a mesh of
one size is another problem for another seed, too.  All outputs are whole
numbers: the colors, the number of rounds and the number of colors.
"""
from __future__ import annotations

import atexit
import math

import numpy as np
import torch

import paper_2107_00075_gb300 as pgc
from paper_2107_00075_gb300 import inputs

_DEV = "cuda"
_FLAGS = {"degree": 0, "no_degree": pgc.PGC_NO_DEGREE_RULE,
          "dynamic": pgc.PGC_PRIORITY_DYNAMIC, "saturation": pgc.PGC_PRIORITY_SATURATION}


def listed():
    return [
        # the smallest member size of the batched workload's decade, as a single call:
        # latency of one call
        {"name": "d1_grid_1000", "call": "d1", "family": "grid", "n": 1000, "rule": "degree"},
        # the 32^3 mesh of the small D1 configuration
        {"name": "d1_mesh7_32", "call": "d1", "family": "mesh", "points": 7,
         "nx": 32, "ny": 32, "nz": 32, "rule": "degree"},
        # an unstructured sparse graph of ordinary size
        {"name": "d1_random_1m", "call": "d1", "family": "random", "n": 1_000_003,
         "degree": 16.0, "rule": "degree"},
        # skewed degrees, ordinary size: long rows and many nearly empty rounds
        {"name": "d1_rmat_20", "call": "d1", "family": "rmat", "n": 1 << 20, "edge_factor": 16,
         "rule": "degree"},
        # the headline configuration: R-MAT scale 24
        {"name": "d1_rmat_24", "call": "d1", "family": "rmat", "n": 1 << 24, "edge_factor": 16,
         "rule": "degree"},
        # the rule whose priorities are recomputed every round (fewest colors)
        {"name": "d1_rmat_18_dynamic", "call": "d1", "family": "rmat", "n": 1 << 18,
         "edge_factor": 16, "rule": "dynamic"},
        # Hessian coloring of a small mesh with uneven sides
        {"name": "d2_mesh7_45x37x31", "call": "d2", "family": "mesh", "points": 7,
         "nx": 45, "ny": 37, "nz": 31, "rule": "degree"},
        # the distance-2 configuration
        {"name": "d2_mesh27_128", "call": "d2", "family": "mesh", "points": 27,
         "nx": 128, "ny": 128, "nz": 128, "rule": "degree"},
        # Jacobian compression, the pattern of the README example
        {"name": "pd2_40k_10k", "call": "pd2", "n_rows": 40_000, "n_cols": 10_000,
         "sides": "columns", "rule": "degree"},
        # the partial distance-2 configuration
        {"name": "pd2_4m_1m", "call": "pd2", "n_rows": 1 << 22, "n_cols": 1 << 20,
         "sides": "columns", "rule": "degree"},
        # the batched configuration: 4096 uneven graphs in one call
        {"name": "batch_4096", "call": "batch", "graphs": 4096, "plan": 1, "rule": "degree"},
        # the server with a full queue, from pinned host memory and back
        {"name": "serve_32", "call": "serve", "requests": 32, "plan": 7},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["d1", "d1", "d1", "d1", "d2", "d2", "pd2", "pd2", "pd2", "batch", "serve"])
    rule = rng.choice(["degree", "degree", "degree", "no_degree"])
    if call == "d1":
        family = rng.choice(["grid", "mesh", "random", "rmat", "rmat"])
        case = {"call": call, "family": family, "rule": rule}
        if family == "grid":
            case["n"] = _log_uniform(rng, 100, 200_000)
        elif family == "mesh":
            case["points"] = rng.choice([7, 27])
            case.update({k: _log_uniform(rng, 8, 160) for k in ("nx", "ny", "nz")})
        elif family == "random":
            case.update(n=_log_uniform(rng, 1000, 1_000_000), degree=round(rng.uniform(2, 32), 2))
        else:
            case.update(n=_log_uniform(rng, 1000, 4_000_000), edge_factor=rng.choice([8, 16]))
            if case["n"] < 300_000 and rng.random() < 0.4:
                case["rule"] = rng.choice(["dynamic", "saturation"])
        return case
    if call == "d2":
        return {"call": call, "family": "mesh", "points": rng.choice([7, 27]), "rule": rule,
                **{k: _log_uniform(rng, 8, 128) for k in ("nx", "ny", "nz")}}
    if call == "pd2":
        sides = rng.choice(["columns", "columns", "both"])
        n_cols = _log_uniform(rng, 200, 1_000_000 if sides == "columns" else 100_000)
        return {"call": call, "n_rows": int(n_cols * rng.uniform(2, 4)), "n_cols": n_cols,
                "sides": sides, "rule": rule}
    if call == "batch":
        return {"call": call, "graphs": _log_uniform(rng, 16, 1024),
                "plan": rng.randrange(1, 1 << 20), "rule": rule}
    return {"call": call, "requests": rng.randrange(4, 33), "plan": rng.randrange(1, 1 << 20)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(seed)
    return g


def _integers(gen, bound, count):
    return (torch.rand(count, generator=gen, device=_DEV, dtype=torch.float64) * bound).long()


def _csr(n, src, dst):
    """Symmetric int32 CSR of undirected samples, repeats and loops dropped."""
    key = torch.cat([src * n + dst, dst * n + src])[torch.cat([src != dst] * 2)]
    key = torch.unique(key)
    row_ptr = torch.searchsorted(key, torch.arange(n + 1, device=_DEV) * n)
    return row_ptr.int(), key.remainder_(n).int()


def _grid(n):
    """2D 5-point grid, ceil(sqrt(n)) columns, last row partial."""
    w = math.isqrt(n - 1) + 1
    v = torch.arange(n, device=_DEV)
    right = v[(v % w != w - 1) & (v + 1 < n)]
    down = v[v + w < n]
    return _csr(n, torch.cat([right, down]), torch.cat([right + 1, down + w]))


def _mesh(nx, ny, nz, points):
    n = nx * ny * nz
    v = torch.arange(n, device=_DEV, dtype=torch.int32)
    x, y, z = v % nx, (v // nx) % ny, v // (nx * ny)
    ids, keep = [], []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                nonzero = abs(dx) + abs(dy) + abs(dz)
                if nonzero == 0 or (points == 7 and nonzero != 1):
                    continue
                ids.append(v + dx + nx * (dy + ny * dz))
                keep.append((x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) &
                            (z + dz >= 0) & (z + dz < nz))
    keep = torch.stack(keep, 1)
    row_ptr = torch.zeros(n + 1, device=_DEV, dtype=torch.int32)
    row_ptr[1:] = keep.sum(1).cumsum(0)
    return row_ptr, torch.stack(ids, 1)[keep]


def _random(n, degree, gen):
    m = round(n * degree / 2)
    return _csr(n, _integers(gen, n, m), _integers(gen, n, m))


def _rmat(n, edge_factor, gen):
    """R-MAT (.57, .19, .19, .05) over the next power of two, ids scrambled;
    samples with an endpoint >= n are drawn again."""
    scale = max(1, math.ceil(math.log2(n)))
    want, srcs, dsts = edge_factor * n, [], []
    while want > 0:
        m = want if n == 1 << scale else 2 * want
        src = torch.zeros(m, device=_DEV, dtype=torch.int64)
        dst = torch.zeros_like(src)
        for _ in range(scale):
            r = torch.rand(m, generator=gen, device=_DEV)
            down = r >= 0.76
            src.mul_(2).add_(down)
            dst.mul_(2).add_(((r >= 0.57) & ~down) | (r >= 0.95))
        src, dst = [(a * 0x9E3779B1 + 12345) & ((1 << scale) - 1) for a in (src, dst)]
        if n < 1 << scale:
            keep = (src < n) & (dst < n)
            src, dst = src[keep][:want], dst[keep][:want]
        srcs.append(src)
        dsts.append(dst)
        want -= src.numel()
    return _csr(n, torch.cat(srcs), torch.cat(dsts))


def _bipartite(n_rows, n_cols, gen):
    """Rows of 1 + Poisson(7) uniform columns, repeats dropped; CSR and CSC."""
    length = 1 + torch.poisson(torch.full((n_rows,), 7.0, device=_DEV), generator=gen).long()
    row = torch.repeat_interleave(torch.arange(n_rows, device=_DEV), length)
    key = torch.unique(row * n_cols + _integers(gen, n_cols, row.numel()))
    row, col = key // n_cols, key % n_cols
    row_ptr = torch.searchsorted(key, torch.arange(n_rows + 1, device=_DEV) * n_cols)
    key = torch.sort(col * n_rows + row)[0]
    col_ptr = torch.searchsorted(key, torch.arange(n_cols + 1, device=_DEV) * n_rows)
    return row_ptr.int(), col.int(), col_ptr.int(), (key % n_rows).int()


def _batch(case, gen):
    """Even members 2D grids, odd members Erdos-Renyi, flattened; edges are
    sorted 256 graphs at a time."""
    sizes, degrees = inputs.batch_plan(case["graphs"], seed=case["plan"])
    n = torch.from_numpy(sizes).to(_DEV)
    vtx_off = torch.zeros(len(sizes) + 1, device=_DEV, dtype=torch.int64)
    vtx_off[1:] = n.cumsum(0)
    row_parts, col_parts, nnz = [], [], [0]
    for lo in range(0, len(sizes), 256):
        part = range(lo, min(lo + 256, len(sizes)))
        first = int(vtx_off[lo])
        srcs, dsts, bases = [], [], []
        odd = [i for i in part if i % 2]
        if odd:
            count = torch.tensor([round(int(sizes[i]) * float(degrees[i]) / 2) for i in odd],
                                 device=_DEV)
            which = torch.repeat_interleave(torch.tensor(odd, device=_DEV), count)
            bound = n[which].double()
            for out in (srcs, dsts):
                out.append((torch.rand(which.numel(), generator=gen, device=_DEV,
                                       dtype=torch.float64) * bound).long())
            bases.append(vtx_off[which] - first)
        even = [i for i in part if i % 2 == 0]
        which = torch.repeat_interleave(torch.tensor(even, device=_DEV), n[even])
        start = vtx_off[:-1][even] - first
        local = torch.arange(which.numel(), device=_DEV)
        local = local - torch.repeat_interleave(n[even].cumsum(0) - n[even], n[even])
        width = torch.repeat_interleave(
            torch.tensor([math.isqrt(int(sizes[i]) - 1) + 1 for i in even], device=_DEV), n[even])
        base = torch.repeat_interleave(start, n[even])
        bound = n[which]
        for step, ok in ((torch.ones_like(width), local % width != width - 1),
                         (width, torch.ones_like(width, dtype=torch.bool))):
            ok = ok & (local + step < bound)
            srcs.append(local[ok])
            dsts.append((local + step)[ok])
            bases.append(base[ok])
        src, dst, base = torch.cat(srcs), torch.cat(dsts), torch.cat(bases)
        ok = src != dst
        src, dst, base = src[ok], dst[ok], base[ok]
        # every local id fits 18 bits (at most 200,000 vertices a graph)
        key = torch.unique(torch.cat([(base + src << 18) | dst, (base + dst << 18) | src]))
        for i in part:
            a, b = int(vtx_off[i]) - first, int(vtx_off[i]) - first + int(sizes[i])
            ends = torch.searchsorted(key, torch.arange(a, b + 1, device=_DEV) << 18)
            row_parts.append((ends - ends[0]).int())
            nnz.append(ends[-1] - ends[0])
        col_parts.append((key & ((1 << 18) - 1)).int())
    nnz_off = torch.stack([torch.as_tensor(x, device=_DEV) for x in nnz]).cumsum(0)
    return vtx_off, nnz_off, torch.cat(row_parts), torch.cat(col_parts)


def _symmetric(case, gen):
    if case["family"] == "grid":
        return _grid(case["n"])
    if case["family"] == "mesh":
        return _mesh(case["nx"], case["ny"], case["nz"], case["points"])
    if case["family"] == "random":
        return _random(case["n"], case["degree"], gen)
    return _rmat(case["n"], case["edge_factor"], gen)


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t).numpy()


def _serve_sizes(case):
    """70% D1 and 30% PD2, vertices log-uniform on [1K, 4M]."""
    rng = np.random.default_rng(case["plan"])
    return [("d1" if rng.random() < 0.7 else "pd2",
             int(math.exp(rng.uniform(math.log(1000), math.log(4_000_000)))))
            for _ in range(case["requests"])]


def _pd2_sides(n):
    return max(1, int(0.8 * n)), max(1, int(0.2 * n))


_server = None


def _the_server():
    """One server for the life of the program, as a service keeps it."""
    global _server
    if _server is None:
        _server = pgc.PgcServer(16 << 30, max_active=16)
        atexit.register(_server.close)
    return _server


def prepare(case, seed):
    gen = _generator(seed)
    state = {"call": case["call"], "seed": seed, "flags": _FLAGS[case.get("rule", "degree")]}
    if case["call"] in ("d1", "d2"):
        state["arrays"] = _symmetric(case, gen)
    elif case["call"] == "pd2":
        state["both"] = case["sides"] == "both"
        state["shape"] = case["n_rows"], case["n_cols"]
        state["arrays"] = _bipartite(case["n_rows"], case["n_cols"], gen)
    elif case["call"] == "batch":
        state["arrays"] = _batch(case, gen)
    else:
        state["server"] = _the_server()
        state["requests"] = []
        for kind, n in _serve_sizes(case):
            if kind == "d1":
                args = tuple(_pinned(a) for a in _rmat(n, 8, gen))
                count = n
            else:
                rows, count = _pd2_sides(n)
                args = (rows, count) + tuple(_pinned(a) for a in _bipartite(rows, count, gen))
            out = torch.zeros(count, dtype=torch.int32, pin_memory=True).numpy()
            state["requests"].append((kind, args, out))
    torch.cuda.synchronize()
    return state


def run(state):
    call, seed = state["call"], state["seed"]
    if call == "serve":
        server = state["server"]
        ids = [(server.submit_d1 if kind == "d1" else server.submit_pd2)(
            *args, seed=seed + i, colors=out)
            for i, (kind, args, out) in enumerate(state["requests"])]
        done = [server.wait(i) for i in ids]
        return ([colors for colors, _ in done],
                np.array([(info.rounds, info.num_colors) for _, info in done]))
    flags = state["flags"]
    if call == "d1":
        r = pgc.pgc_color_d1(*state["arrays"], seed=seed, flags=flags)
    elif call == "d2":
        r = pgc.pgc_color_d2(*state["arrays"], seed=seed, flags=flags)
    elif call == "pd2":
        color = pgc.pgc_color_pd2_bipartite if state["both"] else pgc.pgc_color_pd2
        r = color(*state["shape"], *state["arrays"], seed=seed, flags=flags)
    else:
        r = pgc.pgc_color_d1_batch(*state["arrays"], seed=seed, flags=flags)
        return r.colors, r.rounds_per_graph, r.colors_per_graph, r.rounds
    return r.colors, r.rounds, r.num_colors


def _entries(case):
    """(vertices colored, offsets read, adjacency entries read) of one call;
    repeats among random samples are not taken off."""
    if case["call"] in ("d1", "d2"):
        if case["family"] == "mesh":
            nx, ny, nz = case["nx"], case["ny"], case["nz"]
            n = nx * ny * nz
            if case["points"] == 7:
                nnz = 2 * (3 * n - nx * ny - ny * nz - nx * nz)
            else:
                nnz = (3 * nx - 2) * (3 * ny - 2) * (3 * nz - 2) - n
        else:
            n = case["n"]
            nnz = {"grid": lambda: 4 * n, "random": lambda: n * case["degree"],
                   "rmat": lambda: 2 * n * case["edge_factor"]}[case["family"]]()
        return n, n + 1, nnz
    if case["call"] == "pd2":
        both = case["sides"] == "both"
        return (case["n_cols"] + (case["n_rows"] if both else 0),
                case["n_rows"] + case["n_cols"] + 2, 16 * case["n_rows"])
    if case["call"] == "batch":
        sizes, degrees = inputs.batch_plan(case["graphs"], seed=case["plan"])
        nnz = sum(4 * int(s) if i % 2 == 0 else int(s) * float(d)
                  for i, (s, d) in enumerate(zip(sizes, degrees)))
        return int(sizes.sum()), int(sizes.sum()) + len(sizes), nnz
    total = np.zeros(3)
    for kind, n in _serve_sizes(case):
        if kind == "d1":
            total += (n, n + 1, 16 * n)
        else:
            rows, cols = _pd2_sides(n)
            total += (cols, rows + cols + 2, 16 * rows)
    return tuple(total)


def work(case):
    """Offsets and adjacency read once, colors written once, four bytes each;
    one comparison for each adjacency entry."""
    n, offsets, nnz = _entries(case)
    return {"bytes": float(4 * (n + offsets + nnz)), "flops": float(nnz)}


def exact(case, seed):
    """Outputs are whole numbers, which have to be equal as they are."""
    return None
