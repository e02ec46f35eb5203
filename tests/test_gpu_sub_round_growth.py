"""Where a CTA's sub-rounds stop growing: a hub discovering as many vertices as one CTA keeps
expanding (half its threads and twice its round's items), and one more."""
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


def broom(k, tail):
    """A hub with k out-edges, each the first of a path of `tail` vertices."""
    n = 1 + k * tail
    first = 1 + np.arange(k) * tail
    inner = np.setdiff1d(np.arange(1, n), first + tail - 1)
    return inputs.csr_from_edges(n, np.concatenate([np.zeros(k, int), inner]), np.concatenate([first, inner + 1]),
                                 np.arange(k + inner.size) % 7)


@pytest.mark.parametrize("cta", [128, 256, 512, 1024])
@pytest.mark.parametrize("over", [0, 1])
def test_hub_at_the_bound(ctx, cta, over):
    from paper_1607_05707_gb300 import irgl as C
    from paper_1607_05707_gb300.api import Batch, as_u32

    k = cta // 2 + 2 + over
    g = broom(k, 9)  # ten hops from the hub: one round of fifteen sub-rounds, if the CTA keeps them
    t = dict(cta_size=cta, warp_thresh=1 << 30, cta_thresh=1 << 30, flags=C.IRGL_TUNE_LOCAL(15) | C.IRGL_TUNE_NO_SMEM)
    s = np.array([0], np.uint32)
    dg = ctx.load(g)
    for kind in ("bfs", "sssp"):
        want = oracle.run(kind, g, s)
        out, st = ctx.run(kind, dg, s, tuning=t)
        np.testing.assert_array_equal(as_u32(out)[: g.n], want)
        assert (st["rounds"] > 1) == bool(over)
        b = Batch(ctx)
        b.add(kind, dg, s)
        b.prepare(t)
        b.run()
        np.testing.assert_array_equal(b.result(0)[0], want)
        b.close()
    dg.close()


@pytest.mark.parametrize("flags", [0xF41, 0x101, 0x401])
@pytest.mark.parametrize("cta", [128, 1024])
def test_star_components_fit_the_worklists(ctx, flags, cta):
    # a hub whose label falls again and again, each time pushing every leaf, in a batch of two
    from paper_1607_05707_gb300.api import Batch

    for seed in range(4):
        rng = np.random.default_rng(seed)
        n = int(rng.integers(3000, 9000))
        p = rng.permutation(n)
        u, v = np.full(n - 1, p[0]), p[1:]
        g = inputs.csr_from_edges(n, np.concatenate([u, v]), np.concatenate([v, u]), symmetric=True)
        dg = ctx.load(g)
        want = oracle.cc(n, g.row_ptr, g.col)
        b = Batch(ctx)
        for _ in range(2):
            b.add("cc", dg)
        b.prepare(dict(cta_size=cta, flags=flags))
        for _ in range(20):
            b.run()
            for r in b.results():
                np.testing.assert_array_equal(r, want)
        b.close()
        dg.close()
