"""Near-far SSSP with the sub-rounds it takes by itself: meshes (taken), graphs with a list
at both sides of the threshold (turned off on the host or on the device), limits that no
distance, every distance and single distances reach, overflowing buffers."""
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


class Borrowed:
    """The graph in device arrays of the caller: the host does not know its degrees."""

    def __init__(self, ctx, g):
        import torch
        from paper_1607_05707_gb300 import irgl as C

        self.n = g.n
        self.keep = [torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda() for a in (g.row_ptr, g.col, g.w)]
        torch.cuda.synchronize()
        self.handle = C.irgl_csr_load(ctx.handle, g.n, g.m, *(t.data_ptr() for t in self.keep), C.IRGL_DEVICE_PTRS)

    def close(self):
        from paper_1607_05707_gb300 import irgl as C

        C.irgl_graph_destroy(self.handle)


def with_hub(mesh, deg):
    """The mesh with one vertex of `deg` more out-edges."""
    rng = np.random.default_rng(deg)
    u = np.repeat(np.arange(mesh.n), np.diff(mesh.row_ptr.astype(np.int64)))
    v = mesh.col.astype(np.int64)
    hub = mesh.n // 2
    return inputs.csr_from_edges(mesh.n, np.concatenate([u, np.full(deg, hub)]),
                                 np.concatenate([v, rng.integers(0, mesh.n, size=deg)]),
                                 np.concatenate([mesh.w, rng.integers(0, 100, size=deg)]))


@pytest.mark.parametrize("extra", [0, 20, 31, 40, 3000])
@pytest.mark.parametrize("delta", [1, 97, 1024, 1 << 30])
def test_near_far_sub_rounds(ctx, extra, delta):
    from paper_1607_05707_gb300.api import as_u32

    side = 41 if delta == 1 else 203
    m = inputs.mesh(side, side + 4, seed=extra + 1, del_frac=0.02, extra_frac=0.002, weights=True)
    g = with_hub(m, extra) if extra else m
    s = np.array([3, g.n - 1], np.uint32)
    want = oracle.run("sssp", g, s)
    for dg in (ctx.load(g), Borrowed(ctx, g)):
        for t in (dict(), dict(cta_size=1024), dict(max_blocks=1), dict(cta_size=256, max_blocks=7, flags=1)):
            out, _ = ctx.run("sssp", dg, s, tuning=dict(t, delta=delta, flags=t.get("flags", 0) | 0x40))
            np.testing.assert_array_equal(as_u32(out)[: g.n], want, err_msg=f"{t}")
        dg.close()
