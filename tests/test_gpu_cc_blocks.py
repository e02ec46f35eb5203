"""Pointer-jumping CC over several blocks per CTA (ragged last ones, ids with and without
locality), small dense graphs split into more blocks than 1024 vertices, blocks that are one path."""
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


def check(ctx, n, u, v, **tuning):
    from paper_1607_05707_gb300.api import as_u32

    g = inputs.csr_from_edges(n, np.concatenate([u, v]), np.concatenate([v, u]), symmetric=True)
    dg = ctx.load(g)
    out, _ = ctx.run("cc_jump", dg, tuning=tuning or None)
    np.testing.assert_array_equal(as_u32(out)[:n], oracle.cc(n, g.row_ptr, g.col))
    dg.close()


@pytest.mark.parametrize("n", [40959, 40960, 40961, 155647, 155649, 400_003])
@pytest.mark.parametrize("max_blocks", [0, 1, 3])
@pytest.mark.parametrize("near", [True, False])
def test_blocks_per_cta(ctx, n, max_blocks, near):
    rng = np.random.default_rng(n + max_blocks)
    k = n // 2 + 1 if near else n
    u = rng.integers(0, n, size=k)
    v = np.minimum(u + rng.integers(1, 40, size=k), n - 1) if near else rng.integers(0, n, size=k)
    check(ctx, n, u, v, max_blocks=max_blocks)


@pytest.mark.parametrize("n", [33, 1000, 4096, 8191])
@pytest.mark.parametrize("deg", [8, 17, 60])
def test_small_dense_graphs(ctx, n, deg):
    # half of them in two interleaved components, so that every block holds both
    rng = np.random.default_rng(n + deg)
    u, v = rng.integers(0, n, size=(2, n * deg // 2))
    check(ctx, n, u, v)
    same = (u ^ v) & 1 == 0
    check(ctx, n, u[same], v[same])
    check(ctx, n, u[same], v[same], max_blocks=2, flags=1)


@pytest.mark.parametrize("n", [31, 40960, 40961, 200_001])
def test_paths(ctx, n):
    rng = np.random.default_rng(n)
    ids = np.arange(n)
    for p in (ids, ids[::-1].copy(), rng.permutation(n), np.concatenate([ids[::2], ids[1::2]])):
        check(ctx, n, p[:-1], p[1:])
        check(ctx, n, p[:-1], p[1:], max_blocks=2)
