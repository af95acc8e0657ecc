"""The persistent BF16 trace's hand-over to the FP32 tail: decided once for the whole grid, from the counts before any
block walks the round's pending rays (needs a GPU)."""
import pytest

from paper_2206_10885_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("width", [32, 64])
@pytest.mark.parametrize("tail", [1, 60, 500, 3000, 9000, 96 * 80 * 2])
def test_handover_equals_host_driven_rounds(width, tail):
    """With one evaluation a round, both forms hand over the same rays in the same round, whatever waits in empty
    voxels then: the same image bit for bit, several times over."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2206_10885_gb300 as kns
    desc = S.GridDesc(N=8, sdf_hidden=2, sdf_width=width, col_width=width, occ_res=64)
    with kns.Context(0) as ctx:
        grid = kns.Grid.load(ctx, desc, S.sal_sphere_grid(desc, seed=5))
        try:
            cams = S.orbit_cameras(2, 96, 80, seed=9)

            def render(rounds):
                out = kns.render(ctx, grid, cams, 96, 80, 96, 1e-4, precision=kns.KNS_BF16,
                                 tuning=dict(tail_rays=tail, bf16_inner_steps=1, bf16_rounds=rounds))
                ctx.sync()
                return out
            ref = render(2)
            for _ in range(3):
                out = render(1)
                for k in ref:
                    assert torch.equal(out[k], ref[k]), k
        finally:
            grid.free()
