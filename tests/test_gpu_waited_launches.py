"""Waited-for launches: sources in the kernel's parameters (at most eight) and copied ones,
repeated sources, and the outcome record between asynchronous calls and errors."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1607_05707_gb300 import inputs

pytestmark = pytest.mark.gpu

NO_SMEM, DIROPT, BITMAP, NO_PACKED, DENSE = 0x40, 0x2, 0x4, 0x8, 0x80
LOCAL15 = 15 << 8


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1607_05707_gb300.api import Context

    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("nsrc", [1, 2, 7, 8, 9])
@pytest.mark.parametrize("repeated", [False, True])
def test_sources_in_every_kernel(ctx, nsrc, repeated):
    from paper_1607_05707_gb300.api import as_u32

    rng = np.random.default_rng(nsrc)
    for g in (inputs.rmat(9, 4, seed=3, weights=True), inputs.mesh(37, 90, seed=4, del_frac=0.03, weights=True)):
        dg = ctx.load(g, in_edges=not g.symmetric)
        s = rng.integers(0, g.n, size=nsrc).astype(np.uint32)
        if repeated:
            s[:] = s[rng.integers(0, max(nsrc // 2, 1), size=nsrc)]
        forms = [("bfs", t) for t in (None, dict(flags=NO_SMEM), dict(flags=NO_SMEM | DIROPT), dict(flags=NO_SMEM | BITMAP),
                                      dict(flags=NO_SMEM | DENSE), dict(flags=NO_SMEM | LOCAL15))]
        forms += [("sssp", t) for t in (None, dict(flags=NO_SMEM), dict(flags=NO_SMEM | NO_PACKED), dict(flags=NO_SMEM | DENSE),
                                        dict(flags=NO_SMEM | LOCAL15), dict(flags=NO_SMEM, delta=60),
                                        dict(flags=NO_SMEM | NO_PACKED, delta=60))]
        for kind, t in forms:
            want = oracle.run(kind, g, s)
            out, _ = ctx.run(kind, dg, s, tuning=t)
            np.testing.assert_array_equal(as_u32(out)[: g.n], want, err_msg=f"{kind} {t}")
            np.testing.assert_array_equal(ctx.run_host(kind, dg, s, tuning=t)[0], want, err_msg=f"{kind} {t} host")
        dg.close()


@pytest.mark.parametrize("flags", [0, NO_SMEM])
def test_counters_after_asynchronous_calls_and_errors(ctx, flags):
    from paper_1607_05707_gb300 import irgl as C
    from paper_1607_05707_gb300.api import as_u32

    g = inputs.mesh(30, 31, seed=8)
    dg, s, t, out = ctx.load(g), np.array([5], np.uint32), dict(flags=flags), ctx.state(g.n)
    want = oracle.run("bfs", g, s)
    wl = ctx.worklist(4)
    wl.push(s)

    def run(**kw):
        _, st = ctx.run("bfs", dg, s, out=out, tuning=t, **kw)
        np.testing.assert_array_equal(as_u32(out), want)
        return st

    alone = run()
    assert alone["edges_scanned"] == int(g.out_degree()[want != 0xFFFFFFFF].sum())
    for waited in (run, lambda: ctx.run_host("bfs", dg, s, tuning=t)[1], lambda: ctx.iterate("bfs", dg, wl, out, tuning=t)[1]):
        for k in (1, 3):  # their edges are counted by the next call that waits, once
            for _ in range(k):
                ctx.iterate_async("bfs", dg, wl, out, t)
            st = waited()
            assert (st["edges_scanned"], st["rounds"]) == ((k + 1) * alone["edges_scanned"], alone["rounds"])
        assert waited()["edges_scanned"] == alone["edges_scanned"]
    # an error in a waited-for call, in an asynchronous one read by the next, and in one read by sync
    for fail in (lambda: ctx.run("bfs", dg, s, out=out, tuning=t, max_rounds=2),
                 lambda: ctx.run_host("bfs", dg, s, tuning=t, max_rounds=2),
                 lambda: (ctx.iterate_async("bfs", dg, wl, out, t, max_rounds=2), run()),
                 lambda: (ctx.iterate_async("bfs", dg, wl, out, t, max_rounds=2), ctx.sync())):
        with pytest.raises(C.IrglError) as ei:
            fail()
        assert ei.value.status == C.IRGL_ERR_MAX_ROUNDS
        assert run() == alone
    wl.close()
    dg.close()
