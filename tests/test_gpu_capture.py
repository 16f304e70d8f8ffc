"""V-cycles and their parts inside a caller's stream capture: plain launches only, and the replay's values."""
import ctypes

import numpy as np
import pytest

from synthetic import gauge

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2303_11512_gb300 import api
    return api


def programmatic_edges(graph):
    """Edges of a captured graph that are not plain dependencies (type byte of the edge data)."""
    cu = ctypes.CDLL("libcuda.so.1")
    count = ctypes.c_size_t(0)
    args = [ctypes.c_void_p(graph.raw_cuda_graph()), None, None, None, ctypes.byref(count)]
    assert cu.cuGraphGetEdges_v2(*args) == 0 and count.value > 0
    n = count.value
    nodes = [(ctypes.c_void_p * n)() for _ in range(2)]
    data = (ctypes.c_ubyte * (8 * n))()
    assert cu.cuGraphGetEdges_v2(args[0], *nodes, data, args[4]) == 0
    return sum(data[8 * i + 2] != 0 for i in range(n))


@pytest.mark.parametrize("images", [0, 2, 3])
@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_cycle_in_a_stream_capture(api, images, prec):
    """A V-cycle (FP16 images: with the memset of its 16-bit copy), a sweep and the transfers of a small batch, captured
    after a warm call: no programmatic edge, and a replay on other values gives the bits of plain calls."""
    L, nrhs, pr = 64, 8, getattr(api, prec)
    dt = torch.complex64 if prec == "FP32" else torch.complex128
    s = torch.cuda.Stream()
    ctx = api.Context(s)
    h = api.mg_setup(ctx, torch.from_numpy(gauge.links(gauge.field(L, 3.0, 0, sweeps=10))).cuda(), L, 0.1,
                     tensor_cores=images, seed=1)
    b, x, r = (torch.zeros((nrhs, h.n[0]), dtype=dt, device="cuda") for _ in range(3))
    c = torch.zeros((nrhs, h.n[1]), dtype=dt, device="cuda")

    def calls():
        h.vcycle(0, b, x, pr)
        h.smooth(0, b, x, pr, 1)
        h.restrict(0, x, c, pr)
        h.smooth(1, c, d, pr, 1)
        h.prolong(0, d, r, pr)

    d = torch.zeros_like(c)
    try:
        torch.cuda.synchronize()
        calls()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(g, stream=s):
            calls()
        assert programmatic_edges(g) == 0
        rs = np.random.default_rng(1)
        b.copy_(torch.from_numpy(rs.standard_normal(b.shape) + 1j * rs.standard_normal(b.shape)))
        out = []
        for run in (calls, g.replay):
            d.zero_()
            torch.cuda.synchronize()
            with torch.cuda.stream(s):
                run()
            torch.cuda.synchronize()
            out.append([t.clone() for t in (x, c, d, r)])
        assert all(torch.equal(p, q) for p, q in zip(*out)) and all(t.abs().max() > 0 for t in out[0])
    finally:
        torch.cuda.synchronize()
        h.close()
        ctx.close()
