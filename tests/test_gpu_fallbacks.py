"""The routes taken where memory that the library can do without is refused: results are those of the usual routes, and
what was refused is not asked for on every call (needs a GPU)."""
import numpy as np
import pytest

from paper_2206_10885_gb300 import synth as S
from tests.test_gpu_walk import pack, rays

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def kns():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2206_10885_gb300 as kns
    return kns


@pytest.mark.parametrize("N,res,density", [(4, 8, 0.05), (3, 21, 0.01), (5, 40, 0.2), (5, 40, 1e-3), (4, 128, 1e-4), (2, 2, 0.3)])
def test_walk_without_the_distance_field(kns, N, res, density):
    """Every crossing reaches the voxel and the parameter of the voxel walk, so the results are equal bit for bit."""
    mask = np.random.default_rng(res).random((res,) * 3) < density
    desc = S.GridDesc(N=N, occ_res=res)
    w, words = S.sal_sphere_grid(desc, seed=1), pack(mask)
    o, d = (torch.tensor(v).cuda() for v in rays(4096, np.random.default_rng(1), mask))
    with kns.Context(0) as ctx:
        out = []
        for most in (-1, 0):
            refused = kns.capi.kns_selftest_memory(ctx.handle, most)
            grid = kns.Grid.load(ctx, desc, w, words)
            out.append(kns.trace_rays(ctx, grid, o, d, 64, 1e-4))
            ctx.sync()
            grid.free()
            assert (kns.capi.kns_selftest_memory(ctx.handle, -1) > refused) == (most == 0)
    for k in out[0]:
        assert torch.equal(out[0][k], out[1][k]), k


def test_field_query_without_scratch(kns):
    """Point by point: the same chains for d and the feature; the gradient's sums run in another order."""
    desc = S.config_desc("c1")
    p = torch.rand((40001, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(0)) * 2 - 1
    with kns.Context(0) as ctx:
        grid = kns.Grid.load(ctx, desc, S.sal_sphere_grid(desc, seed=1))
        a = kns.sdf(ctx, grid, p)
        ctx.sync()
        kns.capi.kns_selftest_memory(ctx.handle, 0)
        b = kns.sdf(ctx, grid, p)
        ctx.sync()
        assert kns.capi.kns_selftest_memory(ctx.handle, -1) == 1
        grid.free()
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert float((a[2] - b[2]).abs().max()) < 1e-5


def test_bf16_rounds_without_buckets(kns):
    """Sorted rounds give the same image; the memory is asked for once, and again when there may be room."""
    desc = S.GridDesc(N=8, sdf_hidden=2, sdf_width=32, col_width=32, occ_res=32)
    w, cams = S.sal_sphere_grid(desc, seed=5), S.orbit_cameras(2, 96, 80, seed=3)

    def render():
        out = kns.render(ctx, grid, cams, 96, 80, 96, 1e-4, precision=kns.KNS_BF16, tuning=dict(tail_rays=-1))
        ctx.sync()
        return out
    with kns.Context(0) as ctx:
        grid, other = kns.Grid.load(ctx, desc, w), kns.Grid.load(ctx, desc, w)
        ref = render()
        kns.capi.kns_selftest_memory(ctx.handle, 0)
        outs = [render() for _ in range(3)]
        assert kns.capi.kns_selftest_memory(ctx.handle, 0) == 1
        render()
        other.free()
        outs.append(render())
        assert kns.capi.kns_selftest_memory(ctx.handle, -1) == 3
        outs.append(render())
        grid.free()
    for out in outs:
        for k in ref:
            assert torch.equal(out[k], ref[k]), k


@pytest.mark.parametrize("tail,asked", [(-1, 1), (63, 1), (64, 0), (0, 0)])
def test_a_render_of_no_more_rays_than_the_tail_takes_wants_no_buckets(kns, tail, asked):
    """Its second round is the tail's (tail 0: the default limit, 32,768 rays)."""
    desc = S.GridDesc(N=2, sdf_hidden=2, sdf_width=32, col_width=32)
    with kns.Context(0) as ctx:
        kns.capi.kns_selftest_memory(ctx.handle, 0)
        grid = kns.Grid.load(ctx, desc, S.sal_sphere_grid(desc, seed=5))
        kns.render(ctx, grid, S.orbit_cameras(1, 8, 8, seed=3), 8, 8, 64, 1e-4, precision=kns.KNS_BF16,
                   tuning=dict(tail_rays=tail))
        ctx.sync()
        assert kns.capi.kns_selftest_memory(ctx.handle, -1) == asked
        grid.free()
