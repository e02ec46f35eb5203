"""Long lists that only one CTA meets in a round: its flag for the big phase is not to be lost
whichever warp sets it, however late the thread that starts the round's counters is."""
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


def hubs(n, seed):
    """A sparse random graph whose only long lists are those of three hubs."""
    rng = np.random.default_rng(seed)
    u, v = rng.integers(0, n, size=(2, 2 * n))
    u[:n] = rng.integers(0, n, size=3)[rng.integers(0, 3, size=n)]
    w = rng.integers(0, 101, size=u.size)
    return inputs.csr_from_edges(n, np.concatenate([u, v]), np.concatenate([v, u]), np.concatenate([w, w]), symmetric=True)


@pytest.mark.parametrize("cta", [256, 1024])
def test_hubs_expanded_in_every_run(ctx, cta):
    # a rare loss: about one run in a hundred of the 1024-thread form kept a hub's former distance
    import torch

    rng = np.random.default_rng(cta)
    for n in (9039, 60000):
        g = hubs(n, 5)
        dg = ctx.load(g)
        for kind in ("sssp", "bfs"):
            s = rng.integers(0, n, size=2).astype(np.uint32)
            want = torch.from_numpy(oracle.run(kind, g, s).view(np.int32)).cuda()
            torch.cuda.synchronize()
            out = ctx.state(n)
            for k in range(400):
                ctx.run(kind, dg, s, out=out, tuning=dict(cta_size=cta))
                assert torch.equal(out, want), (kind, k)
        dg.close()


def test_one_hub_in_a_batch(ctx):
    from paper_1607_05707_gb300.api import Batch

    n = 35
    u, v = np.zeros(n - 1, int), np.arange(1, n)
    w = np.random.default_rng(1).integers(0, 101, size=n - 1)
    star = inputs.csr_from_edges(n, np.concatenate([u, v]), np.concatenate([v, u]), np.concatenate([w, w]), symmetric=True)
    rest = inputs.mesh(60, 61, seed=2, weights=True)  # no list for the big phase
    ds, dr = ctx.load(star), ctx.load(rest)
    items = [("sssp", star, ds, [20])] + [("bfs", rest, dr, [k]) for k in range(9)]
    want = [oracle.run(k, g, np.array(s, np.uint32)) for k, g, _, s in items]
    for t in (dict(cta_size=1024), dict(cta_size=1024, flags=0x8)):
        b = Batch(ctx)
        for k, _, d, s in items:
            b.add(k, d, s)
        b.prepare(t)
        for _ in range(300):
            b.run()
            for r, e in zip(b.results(), want):
                np.testing.assert_array_equal(r, e)
        b.close()
    ds.close()
    dr.close()
