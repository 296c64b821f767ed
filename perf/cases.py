"""The library's work as its users have it done, as cases that can be timed and compared.

Every case goes through the package's public calls (`Context.gp_*`) on graphs drawn on the GPU
from a seed.  Graph families, sizes and block counts are those of the benchmark and the tests:
Erdos-Renyi and R-MAT graphs, 2D and 3D grids, up to 2^26 nodes and 671M edges, k from 2 to 300,
unit or random node and edge weights, eps = 0.03.

Kinds of cases (`kind`):
  partition  gp_partition of a device-resident graph: the whole multilevel method
  host       gp_partition_host: the same from page-locked host arrays, block ids back on the host
  batch      gp_partition_batch: many small graphs in one call
  level      one coarsening level through its pieces: gp_coarsen, gp_contract, gp_sparsify, and
             the clustering of the graph they give
  refine     gp_refine of a disturbed partition
  initial    gp_initial_partition of a coarsest graph
  score      gp_project of a coarse partition, gp_cut and gp_modularity of the result
Rows of contracted graphs come in no particular order, so `level` returns the coarse ids and
weights of the input's nodes and the next clustering brought back to them, which depends on
every entry of the contracted and sparsified graphs but not on the order.
"""
from __future__ import annotations

import numpy as np
import torch

import paper_2504_17615_gb300 as gp

EPS = 0.03
MODES = {"tweight": gp.GP_SPARSIFY_TWEIGHT, "uniform": gp.GP_SPARSIFY_UNIFORM,
         "exact": gp.GP_SPARSIFY_TWEIGHT_EXACT}
RMAT_A, RMAT_AB, RMAT_ABC = 0.57, 0.76, 0.95


def listed():
    return [
        # the smallest whole call: a small mesh, where launches and host reads are all there is
        {"name": "partition_grid2d_1k6", "kind": "partition", "family": "grid2d", "nx": 41, "ny": 39,
         "k": 4, "cmax": 1, "wmax": 1},
        # the 65,536-node random graph of the benchmark's smallest configuration
        {"name": "partition_er_64k", "kind": "partition", "family": "er", "n": 65536, "m": 524288,
         "k": 2, "cmax": 1, "wmax": 1},
        # a weighted mesh of ordinary size with ragged sides
        {"name": "partition_grid3d_1m", "kind": "partition", "family": "grid3d", "nx": 101, "ny": 99,
         "nz": 103, "k": 32, "cmax": 3, "wmax": 7},
        # a power-law graph with hubs and isolated nodes at scale (the R-MAT configuration)
        {"name": "partition_rmat_s24", "kind": "partition", "family": "rmat", "scale": 24, "ef": 16,
         "k": 64, "cmax": 1, "wmax": 1},
        # the benchmark's workload: the largest graph, low modularity, sparsification on
        {"name": "partition_er_64m", "kind": "partition", "family": "er", "n": 1 << 26,
         "m": 671088640, "k": 128, "cmax": 1, "wmax": 1},
        # a request from host memory (what a served request does), the benchmark's small workload
        {"name": "host_er_1m", "kind": "host", "family": "er", "n": 1 << 20, "m": 10485760, "k": 128,
         "cmax": 1, "wmax": 1},
        # many small uneven graphs at once (the batched mix)
        {"name": "batch_mix_128", "kind": "batch", "count": 128, "nmin": 1000, "nmax": 100000},
        # one level of the hierarchy on a large random graph, through its pieces
        {"name": "level_er_16m", "kind": "level", "family": "er", "n": 1 << 24, "m": 167772160,
         "k": 128, "cmax": 1, "wmax": 1, "mode": "tweight"},
        # the same on a weighted graph of ordinary odd size with exactly m_hat edges kept
        {"name": "level_er_300k_weighted", "kind": "level", "family": "er", "n": 299993, "m": 3599911,
         "k": 16, "cmax": 5, "wmax": 40, "mode": "exact"},
        # refinement of a projected partition, more blocks than one byte holds
        {"name": "refine_planted_2m_k300", "kind": "refine", "family": "planted", "n": 2000003,
         "m": 16000000, "k": 300, "cmax": 1, "wmax": 1},
        # the coarsest graph of a k = 128 hierarchy
        {"name": "initial_20k_k128", "kind": "initial", "family": "er", "n": 20480, "m": 204800,
         "k": 128, "cmax": 60, "wmax": 30},
        # the value of a partition of a large graph
        {"name": "score_er_8m", "kind": "score", "family": "er", "n": 8388593, "m": 67108864, "k": 64,
         "cmax": 1, "wmax": 1},
    ]


def _log(rng, lo, hi):
    """An integer between lo and hi, spread over its logarithm."""
    return int(round(lo * (hi / lo) ** rng.random()))


def _draw_graph(rng, nmin, nmax, families=("er", "rmat", "grid2d", "grid3d")):
    """A graph of about n nodes, weighted half of the time."""
    n = _log(rng, nmin, nmax)
    fam = rng.choice(families)
    # heavy edges only where the total stays below 2^31 (at most 16 edges a node)
    weights = {"cmax": rng.choice([1, 1, 4]), "wmax": rng.choice([1, 1, 9, 1000] if n < 100000 else [1, 1, 7])}
    if fam in ("er", "planted"):
        return {"family": fam, "n": n, "m": int(n * rng.uniform(4, 16)), **weights}
    if fam == "rmat":
        return {"family": fam, "scale": max(8, n.bit_length() - 1), "ef": rng.choice([8, 16]), **weights}
    if fam == "grid2d":
        nx = max(8, int(n ** 0.5 * rng.uniform(0.5, 2)))
        return {"family": fam, "nx": nx, "ny": max(8, n // nx), **weights}
    nx = max(4, int(n ** (1 / 3) * rng.uniform(0.7, 1.4)))
    ny = max(4, int((n / nx) ** 0.5))
    return {"family": fam, "nx": nx, "ny": ny, "nz": max(4, n // (nx * ny)), **weights}


def draw(rng):
    kind = rng.choice(["partition", "partition", "partition", "host", "batch", "level", "refine", "initial", "score"])
    if kind == "partition":
        return {"kind": kind, **_draw_graph(rng, 2000, 1 << 24), "k": rng.choice([2, 3, 8, 32, 64, 100, 128])}
    if kind == "host":
        return {"kind": kind, **_draw_graph(rng, 2000, 1 << 22), "k": rng.choice([2, 8, 32, 128])}
    if kind == "batch":
        nmin = _log(rng, 1000, 3000)
        return {"kind": kind, "count": rng.randint(16, 160), "nmin": nmin, "nmax": _log(rng, 10000, 100000)}
    if kind == "level":
        return {"kind": kind, **_draw_graph(rng, 20000, 1 << 24), "k": rng.choice([2, 16, 64, 128]),
                "mode": rng.choice(["tweight", "tweight", "uniform", "exact"])}
    if kind == "refine":
        return {"kind": kind, **_draw_graph(rng, 20000, 1 << 23, ("planted", "grid2d", "grid3d")),
                "k": rng.choice([2, 7, 64, 128, 200, 300])}
    if kind == "initial":
        return {"kind": kind, **_draw_graph(rng, 300, 25000, ("er", "grid2d", "grid3d")), "k": rng.choice([2, 5, 64, 128])}
    return {"kind": kind, **_draw_graph(rng, 4000, 1 << 24), "k": rng.choice([2, 64, 255, 300])}


# ----------------------------------------------------------------- graphs

def _pair_weights(lo, hi, wmax, salt):
    """A weight in [1, wmax] per unordered pair: both directions of an edge get the same."""
    x = (lo * 0x9E3779B1 + hi * 0x85EBCA77 + salt * 0xC2B2AE35) & 0x7FFFFFFF
    x = ((x ^ (x >> 15)) * 0x2C1B3C6D) & 0x7FFFFFFF
    x = ((x ^ (x >> 12)) * 0x297A2D39) & 0x7FFFFFFF
    return ((x ^ (x >> 15)) % wmax + 1).to(torch.int32)


def _csr(n, u, v, cmax, wmax, gen, salt):
    """Symmetric CSR with sorted rows of the pairs (u, v), without loops and duplicates."""
    keep = u != v
    u, v = u[keep], v[keep]
    del keep
    key = torch.cat([u * n + v, v * n + u])
    del u, v
    key = torch.sort(key)[0]
    if key.numel():
        first = torch.ones(key.numel(), dtype=torch.bool, device="cuda")
        torch.ne(key[1:], key[:-1], out=first[1:])
        key = key[first]
        del first
    rows = key // n
    xadj = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    xadj[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    m2 = key.numel()
    if wmax > 1:
        cols = key - rows * n
        adjwgt = _pair_weights(torch.minimum(rows, cols), torch.maximum(rows, cols), wmax, salt)
        adjncy = cols.to(torch.int32)
        del cols
    else:
        adjwgt = torch.ones(max(m2, 1), dtype=torch.int32, device="cuda")
        adjncy = (key - rows * n).to(torch.int32)
    del key, rows
    if m2 == 0:
        adjncy = torch.zeros(1, dtype=torch.int32, device="cuda")
        adjwgt = torch.ones(1, dtype=torch.int32, device="cuda")
    if cmax > 1:
        vwgt = torch.randint(1, cmax + 1, (n,), generator=gen, device="cuda", dtype=torch.int32)
    else:
        vwgt = torch.ones(n, dtype=torch.int32, device="cuda")
    return gp.DeviceGraph(n, m2, xadj, adjncy, vwgt, adjwgt)


def _graph(case, seed, gen):
    fam = case["family"]
    if fam == "er":
        n = case["n"]
        u = torch.randint(0, n, (case["m"],), generator=gen, device="cuda")
        v = torch.randint(0, n, (case["m"],), generator=gen, device="cuda")
    elif fam == "planted":  # k communities of consecutive nodes, seven edges of ten inside them
        n, k = case["n"], case["k"]
        size = max(1, n // k)
        u = torch.randint(0, n, (case["m"],), generator=gen, device="cuda")
        v = torch.randint(0, n, (case["m"],), generator=gen, device="cuda")
        inside = torch.rand(case["m"], generator=gen, device="cuda") < 0.7
        v = torch.where(inside, (u // size * size + v % size).clamp_(max=n - 1), v)
    elif fam == "rmat":
        n, m = 1 << case["scale"], case["ef"] << case["scale"]
        u = torch.zeros(m, dtype=torch.int64, device="cuda")
        v = torch.zeros(m, dtype=torch.int64, device="cuda")
        for _ in range(case["scale"]):
            r = torch.rand(m, generator=gen, device="cuda")
            u.mul_(2).add_(r >= RMAT_AB)
            v.mul_(2).add_(((r >= RMAT_A) & (r < RMAT_AB)) | (r >= RMAT_ABC))
            del r
    else:
        nx, ny, nz = case["nx"], case["ny"], case.get("nz", 1)
        n = nx * ny * nz
        x = torch.arange(n, device="cuda")
        right, up, back = x[x % nx < nx - 1], x[x // nx % ny < ny - 1], x[x // (nx * ny) < nz - 1]
        u = torch.cat([right, up, back])
        v = torch.cat([right + 1, up + nx, back + nx * ny])
    return _csr(n, u, v, case["cmax"], case["wmax"], gen, seed & 0xFFFF)


def _batch_graphs(case, seed, gen):
    """The batched mix: n log-uniform, the four families alike often, k in {2 .. 64}."""
    rng = np.random.default_rng((case["count"], case["nmin"], case["nmax"]))  # sizes belong to the case
    jobs = []
    for i in range(case["count"]):
        n = int(round(case["nmin"] * (case["nmax"] / case["nmin"]) ** rng.random()))
        fam = ("er", "grid2d", "grid3d", "rmat")[int(rng.integers(4))]
        c = {"family": fam, "cmax": 1, "wmax": 1}
        if fam == "er":
            c.update(n=n, m=int(n * rng.uniform(4, 16)))
        elif fam == "grid2d":
            nx = max(2, int(n ** 0.5))
            c.update(nx=nx, ny=max(2, n // nx))
        elif fam == "grid3d":
            nx = max(2, int(round(n ** (1 / 3))))
            c.update(nx=nx, ny=nx, nz=max(2, n // (nx * nx)))
        else:
            c.update(scale=max(10, int(round(np.log2(n)))), ef=8)
        jobs.append((_graph(c, seed + i, gen), int(rng.choice([2, 4, 8, 16, 32, 64])), EPS, seed + i))
    return jobs


_ctx = None


def _context():
    """One context for the process, as a program keeps it for all its graphs."""
    global _ctx
    if _ctx is None:
        _ctx = gp.Context(0)
    return _ctx


def prepare(case, seed):
    kind = case["kind"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = {"ctx": _context(), "kind": kind, "k": case.get("k"), "seed": seed}
    if kind == "batch":
        s["jobs"] = _batch_graphs(case, seed, gen)
        return s
    g = s["g"] = _graph(case, seed, gen)
    k = case["k"]
    if kind == "host":
        s["arrays"] = [t.cpu().pin_memory() for t in (g.xadj, g.adjncy, g.vwgt, g.adjwgt)]
        s["n"], s["m2"] = g.n, g.m2
        del s["g"]
    W = int(g.vwgt.sum(dtype=torch.int64))
    if kind == "level":
        s["U"], s["mode"] = max(1, W // (160 * k)), MODES[case["mode"]]
    elif kind == "refine":
        # consecutive ranges as blocks, a fifth of the nodes astray: what projection hands down
        base = (torch.arange(g.n, device="cuda") * k // g.n).to(torch.int32)
        astray = torch.rand(g.n, generator=gen, device="cuda") < 0.2
        rand = torch.randint(0, k, (g.n,), generator=gen, device="cuda", dtype=torch.int32)
        s["blocks"] = torch.where(astray, rand, base).contiguous()
        heaviest = int(torch.zeros(k, dtype=torch.int64, device="cuda").scatter_add_(
            0, s["blocks"].long(), g.vwgt.long()).max())
        s["Lmax"] = max(heaviest, (W + k - 1) // k * 103 // 100)
    elif kind == "score":
        nc = max(k, g.n * 2 // 5)
        s["cmap"] = torch.randint(0, nc, (g.n,), generator=gen, device="cuda", dtype=torch.int32)
        s["coarse"] = torch.randint(0, k, (nc,), generator=gen, device="cuda", dtype=torch.int32)
    return s


def run(s):
    ctx, kind, k, seed = s["ctx"], s["kind"], s["k"], s["seed"]
    if kind == "partition":
        blocks, cut, st = ctx.gp_partition(s["g"], k, EPS, seed)
        return {"blocks": blocks, "cut": cut, "levels": st.levels, "n_coarsest": st.n_coarsest, "ip_cut": st.ip_cut}
    if kind == "host":
        x, a, c, w = s["arrays"]
        blocks, cut, st = ctx.gp_partition_host(s["n"], s["m2"], x, a, c, w, k, EPS, seed)
        return {"blocks": blocks, "cut": cut, "levels": st.levels}
    if kind == "batch":
        res = ctx.gp_partition_batch(s["jobs"], workers=8)
        return {"blocks": torch.cat([b for b, _ in res]), "cuts": np.array([c for _, c in res], dtype=np.int64)}
    g = s["g"]
    if kind == "level":
        cmap, nc, st = ctx.gp_coarsen(g, s["U"], 1, seed)
        coarse = ctx.gp_contract(g, cmap, nc)
        m, mc = g.m2 // 2, coarse.m2 // 2
        m_hat = min(m // 2, m * nc // (2 * g.n))
        nxt, omega = coarse, 0
        if mc > 4 * m_hat:  # the method's trigger (rho = 4)
            nxt, sp = ctx.gp_sparsify(coarse, m_hat, 2, seed, s["mode"])
            omega = sp.omega_t
        cmap2, nc2, st2 = ctx.gp_coarsen(nxt, s["U"], 2, seed)
        weights = ctx.gp_project(cmap, coarse.tensors()[2], g.n)
        upper = ctx.gp_project(cmap, cmap2, g.n)
        return {"cmap": cmap, "weights": weights, "next": upper,
                "counts": [nc, coarse.m2, nxt.m2, omega, nc2, st.lp_moves, st2.lp_moves]}
    if kind == "refine":
        blocks = s["blocks"].clone()  # refined in place; the state keeps the start
        moves = ctx.gp_refine(g, k, s["Lmax"], 1, seed, blocks)
        return {"blocks": blocks, "moves": moves}
    if kind == "initial":
        return {"blocks": ctx.gp_initial_partition(g, k, EPS, seed)}
    fine = ctx.gp_project(s["cmap"], s["coarse"], g.n)
    cut, weights = ctx.gp_cut(g, fine, k)
    mod = ctx.gp_modularity(g, fine, k)
    return {"fine": fine, "cut": cut, "weights": weights, "w_internal": mod.w_internal, "w_total": mod.w_total,
            "q": mod.q, "alpha": mod.alpha, "bound": mod.bound}


def _edges(case):
    """(nodes, CSR entries) of a case's graph, as drawn."""
    fam = case["family"]
    if fam in ("er", "planted"):
        return case["n"], 2 * case["m"]
    if fam == "rmat":
        return 1 << case["scale"], 2 * (case["ef"] << case["scale"])
    nx, ny, nz = case["nx"], case["ny"], case.get("nz", 1)
    return nx * ny * nz, 2 * ((nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1))


def work(case):
    """Each input read once and each output written once (4-byte words); integer work, so no flops."""
    kind = case["kind"]
    if kind == "batch":  # mean n of a log-uniform draw, about 16 entries a node over the families
        lo, hi = case["nmin"], case["nmax"]
        n = case["count"] * ((hi - lo) / np.log(hi / lo) if hi > lo else lo)
        return {"bytes": float(4 * (3 * n + 2 * 10 * n)), "flops": 0}
    n, m2 = _edges(case)
    csr = 2 * n + 2 * m2  # offsets, node weights, ids, edge weights
    if kind == "level":  # the three maps, the coarse offsets and weights, the contracted and the kept entries
        words = csr + 3 * n + 0.4 * n * 5 + 2 * m2 + 0.4 * m2
    elif kind == "score":
        words = csr + 2 * n + 0.4 * n
    elif kind == "refine":
        words = csr + 2 * n
    else:
        words = csr + n
    return {"bytes": float(4 * words), "flops": 0}


def exact(case, seed):
    """The modularity's fractions in 64 bits; all other outputs are whole numbers."""
    if case["kind"] != "score":
        return None
    s = prepare(case, seed)
    g, k = s["g"], s["k"]
    fine = s["coarse"][s["cmap"].long()]
    rows = torch.repeat_interleave(torch.arange(g.n, device="cuda"), (g.xadj[1:] - g.xadj[:-1]).long())
    same = fine[rows] == fine[g.adjncy[:g.m2].long()]
    w = g.adjwgt[:g.m2].long()
    total, inner = int(w.sum()), int((w * same).sum())
    vol = torch.zeros(k, dtype=torch.int64, device="cuda").scatter_add_(0, fine[rows].long(), w)
    weights = torch.zeros(k, dtype=torch.int64, device="cuda").scatter_add_(0, fine.long(), g.vwgt.long())
    share = vol.double() / total if total else vol.double()
    inside = inner / total if total else 0.0
    q, alpha = inside - float((share * share).sum()), float(share.max())
    return {"fine": fine, "cut": (total - inner) // 2, "weights": weights.cpu().numpy(), "w_internal": inner,
            "w_total": total, "q": q, "alpha": alpha, "bound": 1.0 - q - alpha}
