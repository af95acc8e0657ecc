"""Empty-space walks by the distance field, against the oracle's voxel walk: where d is zero everywhere a ray ends at
its entry into the first occupied voxel, so its depth is the walk's result (needs a GPU)."""
import numpy as np
import pytest

import oracle as O
from paper_2206_10885_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def pack(mask):
    bits = np.packbits(mask.reshape(-1), bitorder="little")
    return np.concatenate([bits, np.zeros(-bits.size % 8, np.uint8)]).view(np.uint64)


def rays(n, rng, mask):
    """Rays of unit length from outside and inside the box, some at or near an occupied voxel, one in eight along an
    axis."""
    o = rng.uniform(-1, 1, (n, 3))
    o[: n // 2] *= 2.5 / np.linalg.norm(o[: n // 2], axis=1, keepdims=True)
    to = rng.uniform(-0.9, 0.9, (n, 3))
    at = np.argwhere(mask)[:, ::-1]  # x fastest
    if at.size:
        k = n // 3
        to[::3][:k] = -1 + (at[rng.integers(0, at.shape[0], k)] + rng.uniform(-0.5, 1.5, (k, 3))) * 2.0 / mask.shape[0]
    d = to - o
    d[::8] = np.eye(3)[rng.integers(0, 3, d[::8].shape[0])] * rng.choice([-1.0, 1.0], (d[::8].shape[0], 1))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return o.astype(np.float32), d.astype(np.float32)


@pytest.mark.parametrize("N,res,density", [(4, 8, 0.05), (3, 21, 0.0), (3, 21, 0.01), (5, 40, 0.2), (5, 40, 1e-3),
                                           (4, 128, 1e-4), (4, 128, -1), (2, 2, 0.3)])
def test_walk_reaches_the_first_occupied_voxel(N, res, density):
    """Rays whose result a shift of 2e-3 voxels would move by more than 20 shifts (they pass an edge, or run nearly
    along a face) are left out; for the others an FP32 face parameter is off by less than 20 roundings of a
    coordinate of size 4 a step, 1e-5, and 1e-4 leaves room for the sample's own arithmetic."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2206_10885_gb300 as kns
    rng = np.random.default_rng(res)
    mask = np.zeros((res,) * 3, bool) if density <= 0 else rng.random((res,) * 3) < density
    if density < 0:
        mask[res // 3, res - 1, 5] = True  # one voxel, farther than the field counts from most others
    desc = S.GridDesc(N=N, occ_res=res)
    w, words = np.zeros(desc.n_cells * desc.p_cell, np.float32), pack(mask)
    o, d = rays(4096, rng, mask)
    ref = O.trace_rays(desc, w, words, o, d, 64, 1e-4)["depth"]
    shift = 2e-3 * 2.0 / res
    robust = np.ones(o.shape[0], bool)
    for axis in range(3):
        for sign in (-1, 1):
            t = O.trace_rays(desc, w, words, o.astype(np.float64) + sign * shift * np.eye(3)[axis], d, 64, 1e-4)["depth"]
            with np.errstate(invalid="ignore"):
                robust &= (t == ref) | (np.abs(t - ref) < 20 * shift)
    assert robust.mean() > 0.8
    with kns.Context(0) as ctx:
        grid = kns.Grid.load(ctx, desc, w, words)
        got = kns.trace_rays(ctx, grid, torch.tensor(o).cuda(), torch.tensor(d).cuda(), 64, 1e-4)["depth"]
        ctx.sync()
        got = got.cpu().numpy().astype(np.float64)
        grid.free()
    hit = np.isfinite(ref)
    assert np.array_equal(hit[robust], np.isfinite(got)[robust])
    both = hit & robust
    assert np.all(np.abs(got[both] - ref[both]) < 1e-4)
