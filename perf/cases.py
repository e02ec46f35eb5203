"""The calls a user of the library makes, as measurable cases.

Every case runs one whole query (or one batch, or one burst of served queries) through the
public entry points (:mod:`paper_1607_05707_gb300.api` and the C binding it marshals to).
The graphs are the workload classes of the library: R-MAT power-law graphs (directed,
duplicates and self-loops dropped, weights uniform in [1, 100]) and 4-neighbour meshes, plain or
with a fraction of the edges deleted (1% unless the components are what is asked for) and 0.1% of
the vertices given an extra short-range edge. They are
drawn on the GPU with torch from the seed alone.

A case is a flat dict: ``call`` (run, batch, serve, msf), the graph (``graph``, and ``scale`` /
``ef`` or ``rows`` / ``cols``), the kernel and the launch tuning a user passes (``cta_size``,
``flags``, ``delta``, ...; absent = the library's default).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1607_05707_gb300 import irgl as C
from paper_1607_05707_gb300.api import Batch, Context, Server
from paper_1607_05707_gb300.inputs import CSR

DEV = "cuda:0"
TUNING = ("cta_size", "warp_thresh", "cta_thresh", "flags", "delta", "defer_deg", "defer_delta")
INF = 0xFFFFFFFF
DIROPT = C.IRGL_TUNE_DIROPT
LOCAL15 = C.IRGL_TUNE_LOCAL(15)


# ----------------------------------------------------------------------------- cases

def listed() -> list[dict]:
    return [
        # the smallest calls: a graph of a few thousand vertices, one query, where launches,
        # copies and rounds are all there is (the 64 x 64 grid has 127 levels)
        dict(name="grid64_bfs", call="run", graph="mesh", rows=64, cols=64, deleted=0.0, kernel="bfs", nsrc=1),
        dict(name="rmat10_sssp", call="run", graph="rmat", scale=10, ef=8, kernel="sssp", nsrc=1),
        # an ordinary mid-size query with three sources and default tuning, result wanted on the host
        dict(name="rmat16_bfs_host", call="run", graph="rmat", scale=16, ef=16, kernel="bfs", nsrc=3, host=True),
        # the library's headline graph: BFS direction-optimising (in-edges loaded) and SSSP
        dict(name="rmat20_bfs", call="run", graph="rmat", scale=20, ef=16, kernel="bfs", nsrc=1, in_edges=True,
             cta_size=256, flags=DIROPT),
        dict(name="rmat20_sssp", call="run", graph="rmat", scale=20, ef=16, kernel="sssp", nsrc=1, cta_size=256),
        # a large power-law graph, borrowed from the caller's device arrays, default tuning
        dict(name="rmat23_sssp", call="run", graph="rmat", scale=23, ef=16, kernel="sssp", nsrc=1),
        # road-like meshes: thousands of small frontiers (BFS with CTA-local sub-rounds, SSSP
        # near-far as the library's autotuner picks it) and, on a mesh with one edge in ten
        # missing, connected components by pointer jumping
        dict(name="mesh4096_bfs", call="run", graph="mesh", rows=4096, cols=4096, deleted=0.01, kernel="bfs", nsrc=1,
             flags=LOCAL15),
        dict(name="mesh4096_ccjump", call="run", graph="mesh", rows=4096, cols=4096, deleted=0.1, kernel="cc_jump",
             nsrc=0),
        dict(name="mesh1021_sssp", call="run", graph="mesh", rows=1021, cols=1031, deleted=0.01, kernel="sssp",
             nsrc=1, cta_size=256, delta=1024),
        # batching: 256 multi-source SSSP instances of uneven size in one captured launch, all
        # results fetched with one copy (tuning as the library's autotuner picks it)
        dict(name="batch256_sssp", call="batch", count=256, lo=10, hi=18, ef=8, warp_thresh=64, cta_thresh=512,
             defer_deg=32, defer_delta=4),
        # serving: a burst of 70% BFS / 30% SSSP queries on grids and one R-MAT graph that runs alone
        dict(name="serve96", call="serve", queries=96, grids=12, lo=256, hi=1000, scale=20, ef=16, slots=512,
             epoch_rounds=32, cta_size=1024, flags=DIROPT | LOCAL15, delta=512),
        # minimum spanning forest of a weighted mesh, Atomic ... Else: Retry locks, edges on the device
        dict(name="mesh2048_msf", call="msf", graph="mesh", rows=2048, cols=2048, deleted=0.01, lock="retry"),
    ]


def draw(rng) -> dict:
    """One more case of the same ranges (sizes log-uniform, odd ones among them)."""
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def mesh(lo, hi, missing=None):
        # lo .. hi vertices, sides within a factor of two of each other
        n = logint(lo, hi)
        r = max(2, int(math.sqrt(n * rng.uniform(0.7, 1.4))))
        return dict(graph="mesh", rows=r, cols=max(2, n // r),
                    deleted=round(rng.uniform(*missing), 3) if missing else rng.choice([0.0, 0.01, 0.01]))

    kind = rng.choice(["small", "rmat_bfs", "rmat_sssp", "mesh_bfs", "mesh_sssp", "ccjump", "batch", "serve", "msf"])
    if kind == "small":
        k = rng.choice(["bfs", "sssp", "cc"])
        if k == "cc":
            g = mesh(100, 4000, (0.3, 0.5))
        elif rng.random() < 0.5:
            g = mesh(40, 4000)
        else:
            g = dict(graph="rmat", scale=rng.randint(5, 10), ef=rng.randint(2, 8))
        return dict(call="run", kernel=k, nsrc=0 if k == "cc" else rng.randint(1, 4), host=rng.random() < 0.3, **g)
    if kind == "rmat_bfs":
        c = dict(call="run", graph="rmat", scale=rng.randint(12, 21), ef=rng.randint(4, 16), kernel="bfs",
                 nsrc=rng.randint(1, 12), host=rng.random() < 0.2)
        if rng.random() < 0.6:
            c.update(in_edges=True, flags=DIROPT, cta_size=rng.choice([128, 256]))
        return c
    if kind == "rmat_sssp":
        return dict(call="run", graph="rmat", scale=rng.randint(12, 22), ef=rng.randint(4, 16), kernel="sssp",
                    nsrc=rng.randint(1, 12), cta_size=rng.choice([128, 256]))
    if kind == "mesh_bfs":
        return dict(call="run", kernel="bfs", nsrc=rng.randint(1, 3), flags=rng.choice([LOCAL15, LOCAL15, 0]),
                    **mesh(8_000, 4_000_000))
    if kind == "mesh_sssp":
        return dict(call="run", kernel="sssp", nsrc=1, cta_size=rng.choice([128, 256]), delta=rng.choice([512, 1024, 2048]), **mesh(8_000, 1_000_000))
    if kind == "ccjump":
        return dict(call="run", kernel="cc_jump", nsrc=0, **mesh(8_000, 16_000_000, (0.2, 0.45)))
    if kind == "batch":
        return dict(call="batch", count=logint(8, 200), lo=10, hi=rng.randint(13, 18), ef=8, warp_thresh=64,
                    cta_thresh=512, defer_deg=32, defer_delta=4)
    if kind == "serve":
        return dict(call="serve", queries=logint(8, 90), grids=rng.randint(2, 12), lo=128, hi=rng.randint(256, 1000),
                    scale=rng.randint(15, 20), ef=16, slots=512, epoch_rounds=32, cta_size=1024,
                    flags=DIROPT | LOCAL15, delta=512)
    return dict(call="msf", lock=rng.choice(["blocking", "ticket", "retry"]), **mesh(4_000, 4_000_000))


# ----------------------------------------------------------------------------- inputs (torch only)

def _gen(seed: int, stream: int) -> torch.Generator:
    return torch.Generator(device=DEV).manual_seed((seed * 1_000_003 + stream * 7919 + 12345) % (1 << 62))


def _csr(n: int, key: torch.Tensor, w: torch.Tensor | None) -> dict:
    """CSR (int32 tensors holding uint32 values) from increasing keys u * n + v."""
    u = torch.div(key, n, rounding_mode="floor")
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(u, minlength=n), 0, out=rp[1:])
    col = (key - u * n).to(torch.int32)
    return dict(n=n, m=int(key.numel()), rp=rp.to(torch.int32), col=col, w=w)


def rmat(scale: int, ef: int, seed: int, stream: int = 0) -> dict:
    """R-MAT (.57, .19, .19, .05): ef * 2^scale draws, permuted ids, loops dropped, duplicates merged."""
    gen = _gen(seed, stream)
    n, k = 1 << scale, ef << scale
    u = torch.zeros(k, dtype=torch.int64, device=DEV)
    v = torch.zeros(k, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        r = torch.rand(k, device=DEV, generator=gen)
        hi = r >= 0.76
        u = u * 2 + hi
        v = v * 2 + (((r >= 0.57) & ~hi) | (r >= 0.95))
    perm = torch.randperm(n, device=DEV, generator=gen)
    u, v = perm[u], perm[v]
    key = torch.unique((u * n + v)[u != v])
    w = torch.randint(1, 101, (key.numel(),), dtype=torch.int32, device=DEV, generator=gen)
    return dict(_csr(n, key, w), symmetric=False)


def mesh(rows: int, cols: int, deleted: float, seed: int, stream: int = 0) -> dict:
    """4-neighbour mesh with one weight per undirected edge; "und": each CSR entry's undirected edge."""
    gen = _gen(seed, stream)
    n = rows * cols
    v = torch.arange(n, device=DEV)
    right, down = v[(v % cols) + 1 < cols], v[v < n - cols]
    lo = torch.cat([right, down])
    hi = torch.cat([right + 1, down + cols])
    if deleted > 0:  # edges missing, and 0.1% of the vertices with one short extra edge
        keep = torch.rand(lo.numel(), device=DEV, generator=gen) >= deleted
        k = max(1, round(0.001 * n))
        a = torch.randint(0, n, (k,), device=DEV, generator=gen)
        dr = torch.randint(-8, 9, (k,), device=DEV, generator=gen)
        dc = torch.randint(-8, 9, (k,), device=DEV, generator=gen)
        r, c = torch.div(a, cols, rounding_mode="floor") + dr, a % cols + dc
        ok = (dr.abs() + dc.abs() <= 8) & (r >= 0) & (r < rows) & (c >= 0) & (c < cols) & (dr.abs() + dc.abs() > 0)
        a, b = a[ok], (r * cols + c)[ok]
        lo = torch.cat([lo[keep], torch.minimum(a, b)])
        hi = torch.cat([hi[keep], torch.maximum(a, b)])
    und = torch.unique(lo * n + hi)
    lo = torch.div(und, n, rounding_mode="floor")
    hi = und - lo * n
    wu = torch.randint(1, 101, (und.numel(),), dtype=torch.int32, device=DEV, generator=gen)
    key, order = torch.sort(torch.cat([und, hi * n + lo]))
    most = rows * (cols - 1) + cols * (rows - 1) + max(1, round(0.001 * n))  # whatever the seed deletes
    return dict(_csr(n, key, wu.repeat(2)[order]), symmetric=True, nund=most, und=order % und.numel())


def graph_of(case: dict, seed: int) -> dict:
    if case["graph"] == "rmat":
        return rmat(case["scale"], case["ef"], seed)
    return mesh(case["rows"], case["cols"], case["deleted"], seed)


def sources(g: dict, k: int, seed: int, stream: int = 99) -> np.ndarray:
    """k seeded vertices of out-degree > 0."""
    deg = g["rp"][1:] - g["rp"][:-1]
    have = torch.nonzero(deg > 0).flatten()
    pick = torch.randint(0, have.numel(), (k,), device=DEV, generator=_gen(seed, stream))
    return have[pick].cpu().numpy().astype(np.uint32)


# ----------------------------------------------------------------------------- the user's program

class Borrowed:
    """A graph borrowed from device arrays that the program keeps (no copy, no host check)."""

    def __init__(self, ctx: Context, g: dict, weights: bool):
        flags = C.IRGL_DEVICE_PTRS | (C.IRGL_SYMMETRIC if g["symmetric"] else 0)
        self.n, self.keep = g["n"], g
        self.handle = C.irgl_csr_load(ctx.handle, g["n"], g["m"], g["rp"].data_ptr(), g["col"].data_ptr(),
                                      g["w"].data_ptr() if weights else None, flags)

    def close(self):
        if self.handle:
            C.irgl_graph_destroy(self.handle)
            self.handle = 0


def load(ctx: Context, g: dict, weights: bool, in_edges: bool = False):
    """Host CSR through the library's loader; graphs of over 2^25 edges, and the meshes whose
    symmetry the program vouches for, stay in the device arrays they were made in."""
    if g["m"] > (1 << 25) or g["symmetric"]:
        torch.cuda.current_stream().synchronize()
        return Borrowed(ctx, g, weights)
    host = [g[k].cpu().numpy() if g[k] is not None else None for k in ("rp", "col", "w")]
    return ctx.load(CSR(g["n"], host[0].view(np.uint32), host[1].view(np.uint32), host[2] if weights else None,
                        symmetric=False), in_edges=in_edges)


class State:
    """One program's context, graphs and buffers; closed with it."""

    def __init__(self):
        self.ctx = Context(0, torch.cuda.Stream())
        self.closers = []

    def __del__(self):
        try:
            torch.cuda.synchronize()
            for c in reversed(self.closers):
                c.close()
            self.ctx.close()
        except Exception:
            pass


def tuning_of(case: dict) -> dict | None:
    return {k: case[k] for k in TUNING if k in case} or None


def host_buffer(n: int) -> np.ndarray:
    return torch.zeros(max(n, 1), dtype=torch.int32, pin_memory=True).numpy().view(np.uint32)


def prepare(case: dict, seed: int) -> State:
    s = State()
    s.case, s.tuning = case, tuning_of(case)
    if case["call"] == "run":
        g = graph_of(case, seed)
        s.g = load(s.ctx, g, case["kernel"] == "sssp", case.get("in_edges", False))
        s.closers.append(s.g)
        s.src = sources(g, case["nsrc"], seed) if case["nsrc"] else None
        s.out = host_buffer(g["n"]) if case.get("host") else s.ctx.state(g["n"])
    elif case["call"] == "msf":
        g = graph_of(case, seed)
        s.g = load(s.ctx, g, True)
        s.closers.append(s.g)
        s.und, s.nund = g["und"], g["nund"]
        s.out = torch.empty(max(g["n"] - 1, 1), dtype=torch.int32, device=DEV)
    elif case["call"] == "batch":
        s.batch = Batch(s.ctx)
        for i, (scale, nsrc) in enumerate(instances(case, seed)):
            g = rmat(scale, case["ef"], seed, i)
            dg = Borrowed(s.ctx, g, True)
            s.closers.append(dg)
            s.batch.add("sssp", dg, sources(g, nsrc, seed, 1000 + i))
        s.closers.append(s.batch)
        s.batch.prepare(s.tuning)
        s.out = host_buffer(sum(s.batch.sizes))
    else:
        graphs = []
        for i, q in enumerate(sides(case, seed)):
            graphs.append(mesh(q, q, 0.0, seed, i))
        graphs.append(rmat(case["scale"], case["ef"], seed, 500))
        handles = [load(s.ctx, g, True) for g in graphs[:-1]] + [load(s.ctx, graphs[-1], True, True)]
        s.closers += handles
        # a power-law graph larger than every grid runs its queries alone; else all share the arena
        solo = graphs[-1]["n"] if graphs[-1]["n"] > max(g["n"] for g in graphs[:-1]) else INF
        s.server = Server(s.ctx, arena_bytes=8 << 30, max_slots=case["slots"], epoch_rounds=case["epoch_rounds"],
                          tuning=s.tuning, solo_min_n=solo)
        s.closers.append(s.server)
        # a burst: uniform graphs and 70% BFS (from the case alone, so that every seed's burst has the
        # same size), uniform sources that have an edge
        rng = np.random.default_rng(2006)
        pick = rng.integers(0, len(graphs), size=case["queries"])
        kinds = rng.random(case["queries"]) < 0.7
        offs = np.concatenate([[0], np.cumsum([graphs[i]["n"] for i in pick])])
        s.out = host_buffer(int(offs[-1]))
        s.queries = [("bfs" if kinds[j] else "sssp", handles[i], int(sources(graphs[i], 1, seed, 2000 + j)[0]),
                      s.out[offs[j]:offs[j + 1]]) for j, i in enumerate(pick)]
    torch.cuda.synchronize()
    return s


def instances(case: dict, seed: int):
    """(scale, number of sources) of each instance of a batch: scale uniform in lo..hi, 1-4 sources.
    The scales depend on the case alone, so that every seed's batch has the same size."""
    scales = np.random.default_rng(2004).integers(case["lo"], case["hi"] + 1, size=case["count"])
    nsrcs = np.random.default_rng(seed).integers(1, 5, size=case["count"])
    return [(int(a), int(b)) for a, b in zip(scales, nsrcs)]


def sides(case: dict, seed: int):
    return [int(x) for x in np.random.default_rng(2005).integers(case["lo"], case["hi"] + 1, size=case["grids"])]


def run(s: State):
    call = s.case["call"]
    if call == "run":
        if s.case.get("host"):
            return s.ctx.run_host(s.case["kernel"], s.g, s.src, out=s.out, tuning=s.tuning)[0].view(np.int32)
        return s.ctx.run(s.case["kernel"], s.g, s.src, out=s.out, tuning=s.tuning)[0]
    if call == "batch":
        s.batch.run()
        s.batch.results(s.out)
        return s.out.view(np.int32)
    if call == "serve":
        for kind, g, src, out in s.queries:
            s.server.submit(kind, g, src, out)
        s.server.drain(60.0)
        return s.out.view(np.int32)
    st = C.irgl_msf(s.ctx.handle, s.g.handle, C.IRGL_PERSISTENT, C.LOCKS[s.case["lock"]], s.out.data_ptr(),
                    s.out.numel(), 0, s.tuning)
    # the edges come in no particular order, one direction each: mark the undirected edges taken
    forest = torch.zeros(s.nund, dtype=torch.bool, device=DEV)
    forest[s.und[s.out[:st["edges"]].long()]] = True
    return dict(forest=forest, weight=st["weight"], edges=st["edges"])


# ----------------------------------------------------------------------------- what a pass cannot do without

def size_of(case: dict) -> tuple[int, int]:
    """(vertices, directed edges) of a case's graph, before duplicates and deletions."""
    if case["graph"] == "rmat":
        return 1 << case["scale"], case["ef"] << case["scale"]
    r, c = case["rows"], case["cols"]
    return r * c, 2 * (r * (c - 1) + c * (r - 1))


def work(case: dict) -> dict:
    """Bytes: the CSR read once (offsets, columns, weights where the kernel uses them), the result written once."""
    if case["call"] == "run":
        n, m = size_of(case)
        return dict(bytes=4 * (n + 1) + (8 if case["kernel"] == "sssp" else 4) * m + 4 * n, flops=0)
    if case["call"] == "msf":
        n, m = size_of(case)
        return dict(bytes=4 * (n + 1) + 8 * m + 4 * n, flops=0)
    if case["call"] == "batch":
        v = sum(1 << a for a, _ in instances(case, 0))
        return dict(bytes=v * (4 + 8 * case["ef"] + 4), flops=0)
    # every query reads its graph (30% of them with weights) and writes its result
    sq = [x * x for x in sides(case, 0)]
    per = [4 * n + 4 * n + 4 * n * (4 + 0.3 * 4) for n in sq] + [(1 << case["scale"]) * (8 + case["ef"] * (4 + 0.3 * 4))]
    return dict(bytes=case["queries"] * sum(per) / len(per), flops=0)


# ----------------------------------------------------------------------------- the same answers from plain torch

def relax_to_fixed_point(g: dict, kernel: str, src: np.ndarray | None, limit_rounds: int):
    """Levels, distances or labels in 64 bits by whole-graph relaxation rounds; None past limit_rounds."""
    n = g["n"]
    u = torch.repeat_interleave(torch.arange(n, device=DEV), (g["rp"][1:] - g["rp"][:-1]).long())
    v = g["col"].long()
    if src is None:
        d, step = torch.arange(n, device=DEV), 0
    else:
        d = torch.full((n,), INF, dtype=torch.int64, device=DEV)
        d[torch.from_numpy(src.astype(np.int64)).to(DEV)] = 0
        step = g["w"].long() if kernel == "sssp" else 1
    for _ in range(limit_rounds):
        x = torch.where(d[u] == INF, INF, d[u] + step) if src is not None else d[u]
        e = d.scatter_reduce(0, v, x, "amin")
        if bool((e == d).all()):
            return d
        d = e
    return None


def exact(case: dict, seed: int):
    if case["call"] != "run" or (case["graph"] == "rmat" and case["scale"] > 21):
        return None  # many graphs or a forest: several minutes in plain torch
    g = graph_of(case, seed)
    src = sources(g, case["nsrc"], seed) if case["nsrc"] else None
    d = relax_to_fixed_point(g, case["kernel"], src, 1500 if g["n"] < (1 << 17) else 64)
    if d is None:
        return None  # thousands of rounds over the whole mesh
    d = torch.where(d >= 1 << 31, d - (1 << 32), d)  # the int32 view of the uint32 values
    return d.to(torch.int32).cpu().numpy() if case.get("host") else d.to(torch.int32)
