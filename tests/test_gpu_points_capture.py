"""Field queries under stream capture (needs a GPU)."""
import ctypes as C

import pytest

from paper_2206_10885_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [100, 40001])
def test_captured_query_is_a_graph_of_launches(n):
    """The context's first query is captured (nothing is set up before it).  As a graph without memory of its own it may
    be instantiated twice over, and it is replayed on other points than it was captured with."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2206_10885_gb300 as kns
    cu = C.CDLL("libcuda.so.1")
    vp = C.c_void_p

    def call(name, *args):
        assert getattr(cu, name)(*args) == 0, name
    desc = S.config_desc("c1")
    gen = torch.Generator("cuda").manual_seed(n)
    p, q = (torch.rand((n, 3), device="cuda", generator=gen) * 2 - 1 for _ in range(2))
    with kns.Context(0) as ctx:
        grid = kns.Grid.load(ctx, desc, S.sal_sphere_grid(desc, seed=1))
        stream, pts = torch.cuda.Stream(), p.clone()
        d, f, g = (torch.empty((n, k), device="cuda") for k in (1, 15, 3))
        torch.cuda.synchronize()
        s, graph, execs = vp(stream.cuda_stream), vp(), (vp(), vp())
        call("cuStreamBeginCapture_v2", s, 0)  # CU_STREAM_CAPTURE_MODE_GLOBAL
        kns.capi.kns_sdf(ctx.handle, grid.handle, pts.data_ptr(), n, d.data_ptr(), f.data_ptr(), g.data_ptr(),
                         stream.cuda_stream)
        call("cuStreamEndCapture", s, C.byref(graph))
        for e in execs:
            call("cuGraphInstantiateWithFlags", C.byref(e), graph, C.c_ulonglong(0))
        for e, points in zip(execs, (p, q)):
            pts.copy_(points)
            torch.cuda.synchronize()
            call("cuGraphLaunch", e, s)
            torch.cuda.synchronize()
            ref = kns.sdf(ctx, grid, points)
            ctx.sync()
            # the grouped route's gradient sums run in another order
            assert torch.equal(d[:, 0], ref[0]) and torch.equal(f, ref[1])
            assert float((g - ref[2]).abs().max()) < 1e-5
        for e in execs:
            call("cuGraphExecDestroy", e)
        call("cuGraphDestroy", graph)
        grid.free()
