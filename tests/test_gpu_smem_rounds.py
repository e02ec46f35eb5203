"""The shared-memory Iterate's kinds of round: narrow ones (at most 64 items), four lanes per
item (at most 256), a list per lane (no list above 8 edges), dealt lists; ends inside each."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1607_05707_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1607_05707_gb300.api import Context

    c = Context(0)
    yield c
    c.close()


def both(n, u, v, w=None):
    w = None if w is None else np.concatenate([w, w])
    return inputs.csr_from_edges(n, np.concatenate([u, v]), np.concatenate([v, u]), w, symmetric=True)


def check(ctx, kind, g, s=None, **kw):
    from paper_1607_05707_gb300.api import as_u32

    dg = ctx.load(g)
    out, st = ctx.run(kind, dg, s, **kw)
    np.testing.assert_array_equal(as_u32(out)[: g.n], oracle.run(kind, g, s), err_msg=kind)
    assert st["grid"] == 1
    dg.close()
    return st


@pytest.mark.parametrize("n", [2, 63, 64, 65, 255, 257, 1023, 1024, 1025, 2049, 4000])
@pytest.mark.parametrize("deg", [2, 8, 9])
def test_whole_graph_rounds(ctx, n, deg):
    # every vertex on the first worklist; the longest list has exactly deg entries, if n allows
    rng = np.random.default_rng(n * 10 + deg)
    u, v = np.arange(n - 1), np.arange(1, n)  # a path in id order and one in any order
    p = rng.permutation(n)
    hub, k = n // 2, min(deg - 2, n - 2)
    far = (hub + 2 + np.arange(k)) % n
    far = far[(far != hub) & (far != hub - 1) & (far != hub + 1)]
    u, v = np.concatenate([u, np.full(far.size, hub)]), np.concatenate([v, far])
    w = rng.integers(0, 50, size=u.size)
    for a, b in ((u, v), (p[u], p[v])):
        g = both(n, a, b, w)
        check(ctx, "cc", g)
        check(ctx, "sssp", g, rng.integers(0, n, size=min(n, 700)).astype(np.uint32))


@pytest.mark.parametrize("front", [63, 64, 65, 256, 257, 1024, 1025])
@pytest.mark.parametrize("deg", [7, 8, 9])
def test_frontiers_of_equal_lists(ctx, front, deg):
    # `front` sources of exactly deg out-edges each, every second one reaching the same vertices
    rng = np.random.default_rng(front + deg)
    n = 2 * front + 50
    u = np.repeat(np.arange(front), deg)
    v = rng.integers(front, n, size=u.size)
    v[: u.size // 2] = rng.integers(front, front + 5, size=u.size // 2)
    g = inputs.csr_from_edges(n, u, v, rng.integers(0, 30, size=u.size))
    s = np.arange(front, dtype=np.uint32)
    check(ctx, "bfs", g, s)
    check(ctx, "sssp", g, s)


@pytest.mark.parametrize("levels", [[1, 64, 64, 65, 3], [1, 65, 64, 1, 300, 64, 2], [64, 64, 64], [1, 300, 2000, 5]])
def test_ends_by_max_rounds(ctx, levels):
    from paper_1607_05707_gb300 import irgl as C
    from paper_1607_05707_gb300.api import as_u32

    # layers of the given sizes, each vertex joined to one of the layer before
    off = np.concatenate([[0], np.cumsum(levels)])
    n = int(off[-1])
    u = np.concatenate([off[i] + np.arange(k) % levels[i] for i, k in enumerate(levels[1:])])
    g = inputs.csr_from_edges(n, u, np.arange(levels[0], n))
    s = np.arange(levels[0], dtype=np.uint32)
    want = oracle.run("bfs", g, s)
    dg = ctx.load(g)
    for k in range(1, len(levels) + 2):
        out = ctx.state(n)
        if k >= len(levels):
            _, st = ctx.run("bfs", dg, s, out=out, max_rounds=k)
            assert st["rounds"] == len(levels)
        else:
            with pytest.raises(C.IrglError) as ei:
                ctx.run("bfs", dg, s, out=out, max_rounds=k)
            assert ei.value.status == C.IRGL_ERR_MAX_ROUNDS
        np.testing.assert_array_equal(as_u32(out), np.where(want <= k, want, 0xFFFFFFFF).astype(np.uint32))
    dg.close()
