"""Field queries whose points share few cells (needs a GPU)."""
import pytest

from paper_2206_10885_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def scene():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2206_10885_gb300 as kns
    desc = S.config_desc("c1")
    ctx = kns.Context(0)
    grid = kns.Grid.load(ctx, desc, S.sal_sphere_grid(desc, seed=1))
    yield kns, ctx, grid
    grid.free()
    ctx.close()


def points(n, cells):
    """n points, at random in the first `cells` of a row of 8 cells."""
    p = torch.rand((n, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    return p * torch.tensor([0.25 * cells, 0.25, 0.25], device="cuda") - 1


@pytest.mark.parametrize("n,cells", [(32768, 1), (32783, 1), (40001, 2), (70001, 1), (200000, 3)])
def test_tiles_of_a_few_crowded_cells(scene, n, cells):
    """Every tile of a cell is there, whole and with its remainder: the results are those of single points (the same
    chains for d and the feature; the gradient's sums run in another order)."""
    kns, ctx, grid = scene
    p = points(n, cells)
    a = kns.sdf(ctx, grid, p)
    at = torch.cat([torch.arange(0, n, 97, device="cuda"), torch.arange(n - 40, n, device="cuda")])
    b = kns.sdf(ctx, grid, p[at])  # fewer than are grouped
    ctx.sync()
    assert torch.equal(a[0][at], b[0]) and torch.equal(a[1][at], b[1])
    assert float((a[2][at] - b[2]).abs().max()) < 1e-5
    assert bool(torch.isfinite(a[2]).all())


def test_one_cell_takes_no_longer_than_many(scene):
    """The tiles of one cell are listed in parallel: two million points in one cell were listed by a single thread and
    took several times as long as two million spread over the grid; the same tiles, all else equal, take as long."""
    kns, ctx, grid = scene

    def best(p):
        ms = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            kns.sdf(ctx, grid, p, want_feat=False, want_grad=False)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms[1:])
    n = 2000000
    spread = torch.rand((n, 3), device="cuda") * 2 - 1
    assert best(points(n, 1)) < 1.5 * best(spread)
