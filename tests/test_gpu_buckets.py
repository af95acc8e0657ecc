"""Rounds of the persistent BF16 trace that take their samples from the cells' buckets against rounds driven by
the host, which are always sorted: the same image bit for bit (needs a GPU)."""
import pytest

from paper_2206_10885_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,width", [(1, 32), (2, 32), (2, 64), (8, 32)])
@pytest.mark.parametrize("W,H,cams", [(7, 5, 1), (23, 16, 1), (31, 33, 2), (96, 80, 3)])
def test_bucketed_rounds_equal_sorted_rounds(N, width, W, H, cams):
    """A few cells hold everything: buckets from a handful of samples through one, two and four tiles (128, 256,
    512) to more than a bucket holds (the round is then sorted)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2206_10885_gb300 as kns
    desc = S.GridDesc(N=N, sdf_hidden=2, sdf_width=width, col_width=width, occ_res=32)
    with kns.Context(0) as ctx:
        grid = kns.Grid.load(ctx, desc, S.sal_sphere_grid(desc, seed=5))
        try:
            c = S.orbit_cameras(cams, W, H, seed=W)
            a = [kns.render(ctx, grid, c, W, H, 96, 1e-4, precision=kns.KNS_BF16, tuning=dict(tail_rays=-1, **t))
                 for t in (dict(), dict(bf16_inner_steps=1), dict(bf16_rounds=2))]
            ctx.sync()
        finally:
            grid.free()
    for k in a[0]:
        assert torch.equal(a[0][k], a[2][k]) and torch.equal(a[1][k], a[2][k]), k
