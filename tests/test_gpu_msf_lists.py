"""Minimum spanning forest at the sizes where its staged lists and its pointer jumping
change: worklists around one stage of the smallest and largest CTAs, and chains (a path
of rising weights hooks into one tree as deep as the path) around the jump's step bound."""
from __future__ import annotations

import numpy as np
import pytest

from test_gpu_msf import check, ctx, sym  # noqa: F401  (ctx: the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [63, 64, 65, 66, 129, 543, 545, 4097, 20011])
def test_chains_and_stages(ctx, n):  # noqa: F811
    path = sym(n, np.arange(n - 1), np.arange(1, n), np.arange(n - 1) % (1 << 20))
    falling = sym(n, np.arange(n - 1), np.arange(1, n), np.arange(n - 1)[::-1] % (1 << 20))
    rng = np.random.default_rng(n)
    u, v = rng.integers(0, n, size=3 * n), rng.integers(0, n, size=3 * n)
    ties = sym(n, u, v, rng.integers(0, 2, size=3 * n))  # equal prefixes decided by the larger end
    for g in (path, falling, ties):
        dg = ctx.load(g)
        for lock in ("blocking", "ticket", "retry"):
            check(ctx, g, dg, "persistent", lock, dict(cta_size=128, max_blocks=2))
            check(ctx, g, dg, "persistent", lock, dict(cta_size=1024))
        check(ctx, g, dg, "per_launch", "retry", dict(cta_size=256))
        dg.close()


@pytest.mark.parametrize("lock", ["blocking", "ticket", "retry"])
@pytest.mark.parametrize("mode", ["persistent", "per_launch"])
def test_locks_counted_only_where_taken(ctx, lock, mode):
    n = 5000
    # pairs: the forest is complete after the first iteration, in which no component is shared;
    # a path of alternating weights is pairs after it, and takes more iterations
    pairs = sym(n, np.arange(0, n, 2), np.arange(1, n, 2), np.arange(n // 2) % 9)
    path = sym(n, np.arange(n - 1), np.arange(1, n), np.arange(n - 1) % 2)
    for g, locked in ((pairs, False), (path, True)):
        dg = ctx.load(g)
        _, st = ctx.msf(dg, mode=mode, lock=lock)
        assert (st["locks"] > 0) == locked
        assert st["edges"] == (n - 1 if locked else n // 2)
        dg.close()
