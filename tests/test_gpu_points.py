"""The batch field query's two routes -- one point per warp, and points grouped by cell -- against the oracle
at the sizes where they change over, with every combination of outputs (needs a GPU)."""
import numpy as np
import pytest

import oracle as O
from paper_2206_10885_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def kns():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2206_10885_gb300 as kns
    return kns


@pytest.mark.parametrize("width,hidden,L", [(32, 2, 4), (64, 3, 6)])
@pytest.mark.parametrize("n", [1, 5, 32767, 32768, 40001])
def test_points_routes_match_oracle(kns, width, hidden, L, n):
    """8^3 cells: 32,768 points are the first that are grouped (64 a cell, ragged tiles of 16)."""
    desc = S.GridDesc(N=8, sdf_hidden=hidden, sdf_width=width, col_width=width, pe_pos_L=L, pe_dir_L=2 if L == 4 else 4)
    w = S.sal_sphere_grid(desc, seed=4)
    pts = S.uniform_points(n, seed=n, lo=-1.1, hi=1.1)  # points outside the box take the nearest cell
    pts[: n // 3] = pts[0] + np.float32(1e-3) * pts[: n // 3]  # a third of them in a cell or two
    with kns.Context(0) as ctx:
        grid = kns.Grid.load(ctx, desc, w)
        try:
            p = torch.from_numpy(pts).cuda()
            outs = [kns.sdf(ctx, grid, p, f, g) for f, g in ((True, True), (True, False), (False, True), (False, False))]
            ctx.sync()
        finally:
            grid.free()
    od, of, og, _ = O.sdf(desc, w, pts.astype(np.float64))
    for (d, f, g), name in zip(outs, ("all", "feature", "gradient", "d")):
        # FP32 sums of up to 64 terms of order 1 through 4 layers, as the parity suite allows; the gradient
        # grows by 2^(L-1) pi through the encoding
        assert np.max(np.abs(d.cpu().numpy() - od)) < 2e-6, name
        if f is not None:
            assert np.max(np.abs(f.cpu().numpy() - of)) < 5e-6, name
        if g is not None:
            assert np.max(np.abs(g.cpu().numpy() - og)) < 1e-4 * (1 if L == 4 else 4), name


def test_points_in_several_chunks(kns):
    """More points than are grouped at a time (4,194,304): the rest of the batch lands behind the first chunk."""
    desc = S.config_desc("c1")
    w = S.sal_sphere_grid(desc, seed=1)
    n = (1 << 22) + 37
    p = torch.rand((n, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(0)) * 2 - 1
    with kns.Context(0) as ctx:
        grid = kns.Grid.load(ctx, desc, w)
        try:
            d, f, g = kns.sdf(ctx, grid, p)
            at = torch.tensor([0, 1, (1 << 22) - 1, 1 << 22, n - 1], device="cuda")
            ds, fs, gs = kns.sdf(ctx, grid, p[at])
            ctx.sync()
        finally:
            grid.free()
    # the two routes form d and the feature by the same chains; the gradient's sums run in another order
    assert torch.equal(d[at], ds) and torch.equal(f[at], fs)
    assert float((g[at] - gs).abs().max()) < 1e-5
