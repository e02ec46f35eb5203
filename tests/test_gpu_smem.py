"""The shared-memory Iterate at its frontier and list bounds: frontiers on both sides of
four lanes per item (256) and of one item per thread (1024), lists of 4, 5, 32 and 33 edges."""
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


@pytest.mark.parametrize("front", [1, 31, 32, 255, 256, 257, 1023, 1024, 1025])
@pytest.mark.parametrize("deg", [1, 4, 5, 32, 33])
def test_frontiers_and_lists(ctx, front, deg):
    from paper_1607_05707_gb300.api import as_u32

    # a hub reaching `front` vertices at once, each with `deg` edges (bounded by the shared memory)
    rng = np.random.default_rng(front * 100 + deg)
    n = front + 1 + min(front, 500)
    k = min(front, 9000 // deg)
    u = np.concatenate([np.zeros(front, int), np.repeat(np.arange(1, k + 1), deg)])
    v = np.concatenate([np.arange(1, front + 1), rng.integers(0, n, size=k * deg)])
    g = inputs.csr_from_edges(n, u, v, rng.integers(0, 100, size=u.size))
    sym = inputs.csr_from_edges(n, np.concatenate([u, v]), np.concatenate([v, u]), symmetric=True)
    for kind, graph, srcs in (("bfs", g, [0]), ("sssp", g, [0, n - 1, 0]), ("cc", sym, None)):
        dg = ctx.load(graph)
        s = None if srcs is None else np.array(srcs, np.uint32)
        out, st = ctx.run(kind, dg, s)
        np.testing.assert_array_equal(as_u32(out)[:n], oracle.run(kind, graph, s), err_msg=kind)
        assert st["grid"] == 1
        dg.close()
