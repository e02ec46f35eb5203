"""Sparse rounds with CTA-local sub-rounds where their buffers and lists change: halves of
the stage that overflow, lists at both sides of four lanes / one warp / the whole grid,
and batches that mix BFS, SSSP and CC with and without near-far."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1607_05707_gb300 import inputs

pytestmark = pytest.mark.gpu

NO_SPLIT, NO_SMEM = 0x1, 0x40


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1607_05707_gb300.api import Context

    c = Context(0)
    yield c
    c.close()


def bursts(seed, deg, symmetric=False):
    """A chain of hubs, each with `deg` leaves that meet at the next hub, and random chords."""
    rng = np.random.default_rng(seed)
    hubs = 5
    n = hubs * (deg + 1) + 1
    first = np.arange(hubs) * (deg + 1)
    leaves = first[:, None] + 1 + np.arange(deg)
    u = np.concatenate([np.repeat(first, deg), leaves.ravel(), rng.integers(0, n, size=n // 2)])
    v = np.concatenate([leaves.ravel(), np.repeat(first + deg + 1, deg), rng.integers(0, n, size=n // 2)])
    w = rng.integers(0, 50, size=u.size)
    if symmetric:
        u, v, w = np.concatenate([u, v]), np.concatenate([v, u]), np.concatenate([w, w])
    return inputs.csr_from_edges(n, u, v, w, symmetric=symmetric)


@pytest.mark.parametrize("deg", [3, 4, 5, 31, 32, 33, 400, 6000])
def test_lists_and_overflow(ctx, deg):
    from paper_1607_05707_gb300.api import as_u32

    g = bursts(deg, deg)
    dg = ctx.load(g)
    for k, cta, extra in ((15, 128, 0), (15, 1024, NO_SPLIT), (1, 256, NO_SPLIT), (4, 512, 0)):
        for srcs in ([0], [0, 7, 0]):
            s = np.array(srcs, np.uint32)
            for kind in ("bfs", "sssp"):
                for grid in (0, 1, 2):
                    t = dict(cta_size=cta, flags=(k << 8) | extra | NO_SMEM, max_blocks=grid)
                    out, _ = ctx.run(kind, dg, s, tuning=t)
                    np.testing.assert_array_equal(as_u32(out)[: g.n], oracle.run(kind, g, s), err_msg=f"{kind} {t}")
    dg.close()


@pytest.mark.parametrize("delta", [0, 16, 400])
@pytest.mark.parametrize("cta", [128, 1024])
def test_mixed_batches(ctx, delta, cta):
    from paper_1607_05707_gb300.api import Batch

    graphs = [bursts(1, 40, True), inputs.mesh(60, 71, seed=2, del_frac=0.02, extra_frac=0.01, weights=True),
              bursts(3, 3000, True)]
    handles = [ctx.load(g) for g in graphs]
    for k in (0, 3, 15):
        b = Batch(ctx)
        asked = []
        for j in range(30):
            i, kind = j % 3, ("bfs", "sssp", "sssp", "cc")[j % 4]
            s = None if kind == "cc" else np.array([(37 * j) % graphs[i].n], np.uint32)
            b.add(kind, handles[i], s)
            asked.append((kind, graphs[i], s))
        b.prepare(dict(cta_size=cta, flags=k << 8, delta=delta, max_blocks=0 if k == 3 else 4))
        b.run()
        b.run()
        for got, (kind, g, s) in zip(b.results(), asked):
            np.testing.assert_array_equal(got, oracle.run(kind, g, s), err_msg=f"{kind} k={k}")
        b.close()
    for h in handles:
        h.close()


@pytest.mark.parametrize("k", [0, 1, 15])
def test_server_first_epoch_isolated_source(ctx, k):
    # a query that never pushes, admitted in a server's first epoch
    from paper_1607_05707_gb300.api import Server

    g = inputs.csr_from_edges(50, [1, 2], [2, 3], [4, 5])
    dg = ctx.load(g)
    for kind in ("sssp", "bfs"):
        srv = Server(ctx, arena_bytes=1 << 20, max_slots=4, epoch_rounds=8, tuning=dict(flags=k << 8), solo_min_n=0xFFFFFFFF)
        out = np.zeros(50, np.uint32)
        t = srv.submit(kind, dg, 7, out)
        srv.drain(10.0)
        assert srv.poll(t)["status"] == 0
        np.testing.assert_array_equal(out, oracle.run(kind, g, np.array([7], np.uint32)))
        srv.close()
    dg.close()
