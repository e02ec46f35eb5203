"""Worklists of near-far SSSP's sub-rounds: what they take, and the call without them."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1607_05707_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1607_05707_gb300.api import Context

    c = Context(0)
    yield c
    c.close()


def test_memory_of_a_near_far_call(ctx):
    import torch

    from paper_1607_05707_gb300.api import as_u32

    g = inputs.mesh(1024, 1024, seed=5, del_frac=0.01, extra_frac=0.001, weights=True)
    dg, s, out = ctx.load(g, validate=False), np.array([77], np.uint32), ctx.state(g.n)
    # two-array distances: every list the call needs but the packed words and the sub-rounds' own
    ctx.run("sssp", dg, s, out=out, tuning=dict(delta=1024, flags=0x8))
    before = torch.cuda.mem_get_info()[0]
    _, st = ctx.run("sssp", dg, s, out=out, tuning=dict(delta=1024))
    grown = before - torch.cuda.mem_get_info()[0]
    # 8 bytes a vertex for the packed words, two lists of at most 4 n entries, allocator granularity
    assert grown <= 8 * g.n + 2 * 4 * 4 * g.n + (8 << 20)
    np.testing.assert_array_equal(as_u32(out), oracle.run("sssp", g, s))
    dg.close()


@pytest.mark.parametrize("delta", [97, 1024])
def test_lists_refused(ctx, delta):
    from paper_1607_05707_gb300.api import as_u32

    g = inputs.mesh(203, 207, seed=6, del_frac=0.02, extra_frac=0.002, weights=True)
    dg, s = ctx.load(g), np.array([3, g.n - 1], np.uint32)
    want = oracle.run("sssp", g, s)
    ctx.debug_set(9, 1)
    out, plain = ctx.run("sssp", dg, s, tuning=dict(delta=delta))
    np.testing.assert_array_equal(as_u32(out)[: g.n], want)
    ctx.debug_set(9, 0)
    out, own = ctx.run("sssp", dg, s, tuning=dict(delta=delta))  # asked for again: nothing was refused by the device
    np.testing.assert_array_equal(as_u32(out)[: g.n], want)
    assert own["rounds"] < plain["rounds"]
    ctx.debug_set(9, 1)  # lists in hand stay in use
    out, kept = ctx.run("sssp", dg, s, tuning=dict(delta=delta))
    np.testing.assert_array_equal(as_u32(out)[: g.n], want)
    assert kept["rounds"] < plain["rounds"]
    dg.close()
