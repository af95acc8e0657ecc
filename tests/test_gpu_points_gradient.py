"""The field query's gradient where softplus is nearly flat (needs a GPU)."""
import numpy as np
import pytest

import oracle as O
from paper_2206_10885_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("width,hidden", [(32, 2), (32, 3), (64, 2), (64, 3)])
@pytest.mark.parametrize("n", [257, 40001])
def test_gradient_of_units_far_below_zero(width, hidden, n):
    """Every unit's sum lies between -0.33 and -0.2, where softplus' is 5e-15 to 2e-9 and 1 + e^(beta s) rounds to 1.  All
    weights are positive, so nothing cancels and errors are relative: three roundings of a sum of size 0.33, times beta =
    100, are 1e-5 of a unit's slope, the fast exponential at arguments of 33 adds 3e-6 and a sum of 64 terms 4e-6; three
    layers of that stay below 1e-4.  (Softplus itself is lost to FP32 here, 2e-11 at most: the hidden weights are small
    enough for the next sums not to notice.)"""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2206_10885_gb300 as kns
    desc = S.GridDesc(N=4, sdf_hidden=hidden, sdf_width=width, col_width=width)
    rng = np.random.default_rng(width + hidden)
    w = np.zeros((desc.n_cells, desc.p_cell))
    offs, ns = S.layer_offsets(desc), len(desc.sdf_layers())
    for li in range(ns):
        wo, bo, nin, nout = offs[li]
        W = rng.uniform(0.1, 1, (desc.n_cells, nout, nin))
        if li == 0:  # x alone: the sums stay within 0.03 of the bias
            W[:, :, :3] *= 0.01
            W[:, :, 3:] = 0.0
        else:
            W *= 1e4 / nin if li + 1 < ns else 1e16
        w[:, wo:bo] = W.reshape(desc.n_cells, -1)
        w[:, bo:bo + nout] = rng.uniform(-0.3, -0.22, (desc.n_cells, nout)) if li + 1 < ns else 0.0
    w = w.astype(np.float32).reshape(-1)
    pts = S.uniform_points(n, seed=n)
    with kns.Context(0) as ctx:
        grid = kns.Grid.load(ctx, desc, w)
        g = kns.sdf(ctx, grid, torch.from_numpy(pts).cuda())[2]
        ctx.sync()
        grid.free()
    ref = O.sdf(desc, w, pts.astype(np.float64))[2]
    assert ref.min() > 0 and np.max(np.abs(g.cpu().numpy() / ref - 1)) < 1e-4
