"""Where an FP32 render's rounds end: the number of rounds the host launches depends on how many rays each
round holds against the tail's limit and on the rays waiting in empty voxels; the image does not (needs a GPU)."""
import numpy as np
import pytest

from paper_2206_10885_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def scene():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2206_10885_gb300 as kns
    desc = S.config_desc("c2")  # with an occupancy mask: rays wait in empty voxels between rounds
    ctx = kns.Context(0)
    grid = kns.Grid.load(ctx, desc, S.sal_sphere_grid(desc))
    cams = S.orbit_cameras(2, 96, 64, seed=3)
    ref = kns.render(ctx, grid, cams, 96, 64, 128, 1e-4, tuning=dict(tail_rays=-1))  # rounds to the last ray
    ctx.sync()
    yield kns, ctx, grid, cams, ref
    grid.free()
    ctx.close()


@pytest.mark.parametrize("block_tiles", [0, 2, 3])
@pytest.mark.parametrize("tail", [1, 7, 300, 2 * 96 * 64 - 1, 2 * 96 * 64, 2 * 96 * 64 + 1])
def test_last_round_for_any_tail_limit(scene, tail, block_tiles):
    kns, ctx, grid, cams, ref = scene
    out = kns.render(ctx, grid, cams, 96, 64, 128, 1e-4, tuning=dict(tail_rays=tail, block_tiles=block_tiles))
    ctx.sync()
    for k in ref:
        assert torch.equal(out[k], ref[k]), k
    trace = ctx.round_trace()
    assert trace[0]["live"] > 0 and all(r["live"] >= 0 for r in trace)
    if tail >= 2 * 96 * 64:
        assert len(trace) == 1  # no more rays than the tail takes: one round, nothing read by the host


def test_step_budget_ends_the_rounds(scene):
    """One step and a few: rays leave by the budget in the first rounds."""
    kns, ctx, grid, cams, _ = scene
    for steps in (1, 2, 5):
        a = kns.render(ctx, grid, cams, 96, 64, steps, 1e-4)
        b = kns.render(ctx, grid, cams, 96, 64, steps, 1e-4, tuning=dict(tail_rays=-1))
        ctx.sync()
        for k in a:
            assert torch.equal(a[k], b[k]), (steps, k)


@pytest.mark.parametrize("width", [32, 64])
@pytest.mark.parametrize("W,H", [(1, 1), (17, 1), (33, 4), (129, 3), (160, 96)])
def test_warp_private_tiles(width, W, H):
    """The default evaluator against the one whose blocks share their tiles: every sample is the same sum, so the
    images are equal bit for bit, whatever the tile's remainder and however long a warp stays in a cell."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2206_10885_gb300 as kns
    with kns.Context(0) as ctx:
        for res in (0, 64):
            desc = S.GridDesc(N=4, sdf_width=width, col_width=width, pe_pos_L=4 if width == 32 else 6,
                              pe_dir_L=2 if width == 32 else 4, occ_res=res)
            grid = kns.Grid.load(ctx, desc, S.sal_sphere_grid(desc))
            cams = S.orbit_cameras(1, W, H, seed=7)
            ref = kns.render(ctx, grid, cams, W, H, 64, 1e-4, tuning=dict(tail_rays=-1, block_tiles=1))
            for tune in (dict(), dict(inner_steps=1), dict(inner_steps=64, min_active=1), dict(min_active=128)):
                out = kns.render(ctx, grid, cams, W, H, 64, 1e-4, tuning=dict(tail_rays=-1, block_tiles=4, **tune))
                ctx.sync()
                for k in ref:
                    assert torch.equal(out[k], ref[k]), (res, tune, k)
            grid.free()
