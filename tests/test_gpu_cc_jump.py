"""Pointer-jumping CC at the sizes where its blocks, lists and passes change:
one block and a ragged last one, ids with and without locality, lists at both
sides of the lane / warp / whole-grid bounds, a full big list, unsorted rows."""
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


def symmetric(n, u, v, shuffle=None):
    g = inputs.csr_from_edges(n, np.concatenate([u, v]), np.concatenate([v, u]), symmetric=True)
    if shuffle is not None:  # rows in any order
        row = np.repeat(np.arange(n), np.diff(g.row_ptr.astype(np.int64)))
        g.col = g.col[np.lexsort((shuffle.random(g.m), row))]
    return g


def check(ctx, g, tuning=None):
    from paper_1607_05707_gb300.api import as_u32

    dg = ctx.load(g)
    out, st = ctx.run("cc_jump", dg, tuning=tuning)
    np.testing.assert_array_equal(as_u32(out)[: g.n], oracle.cc(g.n, g.row_ptr, g.col))
    assert st["edges_scanned"] == g.m
    dg.close()


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1023, 1024, 1025, 155647, 155649, 400_003])
@pytest.mark.parametrize("near", [True, False])
def test_block_edges(ctx, n, near):
    rng = np.random.default_rng(n)
    k = n // 2 + 1 if near else n
    u = rng.integers(0, n, size=k)
    v = np.minimum(u + rng.integers(1, 40, size=k), n - 1) if near else rng.integers(0, n, size=k)
    check(ctx, symmetric(n, u, v, rng), None if n % 2 else dict(max_blocks=3))


@pytest.mark.parametrize("deg", [15, 16, 17, 511, 512, 513, 5000])
def test_list_bounds(ctx, deg):
    # hubs of exactly deg entries over shuffled ids, in several components
    rng = np.random.default_rng(deg)
    hubs, n = 6, 6 * (deg + 1) + 40
    ids = rng.permutation(n)
    u = np.repeat(ids[:hubs], deg)
    v = ids[hubs:hubs + hubs * deg]
    g = symmetric(n, u, v, rng)
    assert int(g.out_degree().max()) == deg
    for tuning in (None, dict(flags=1), dict(cta_thresh=1 << 30, warp_thresh=1 << 30)):
        check(ctx, g, tuning)
    ctx.debug_set(4, 2)  # a big list of two entries: the other hubs are walked by a warp
    try:
        check(ctx, g)
    finally:
        ctx.debug_set(4, 0)


def test_max_rounds(ctx):
    from paper_1607_05707_gb300 import irgl as C

    g = symmetric(10, np.array([1, 2, 8]), np.array([2, 3, 9]))
    dg = ctx.load(g)
    with pytest.raises(C.IrglError) as ei:
        ctx.run("cc_jump", dg, max_rounds=1)
    assert ei.value.status == C.IRGL_ERR_MAX_ROUNDS
    out, _ = ctx.run("cc_jump", dg, max_rounds=2)
    np.testing.assert_array_equal(out.cpu().numpy()[:10], [0, 1, 1, 1, 4, 5, 6, 7, 8, 8])
    dg.close()
