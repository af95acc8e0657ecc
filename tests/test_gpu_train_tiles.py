"""The training kernels' warp tiles and chunks at their edges against the FP64 oracle (needs a GPU)."""
import numpy as np
import pytest

import oracle
from paper_2206_10885_gb300 import synth as S
from tests.test_gpu_train import assert_grad_close, desc_of, gpu_batch, oracle_args, problem, train_weights

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("H", [2, 3])
@pytest.mark.parametrize("B,Ns,M", [(1, 2, 1), (5, 3, 2), (16, 2, 11), (17, 2, 0), (43, 16, 0), (129, 5, 37), (260, 16, 9)])
def test_one_cell_with_ragged_tiles_and_chunks(H, B, Ns, M):
    """A one-cell grid: every record falls into the same chunks, so the record counts are the tile and chunk
    sizes -- a few records, tiles of 16 and 32 with and without remainders, chunks of 4,096 crossed."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2206_10885_gb300 as kns
    desc = desc_of(1, H)
    w = train_weights(desc, seed=11)
    pr = problem(desc, B, Ns, 1, max(M, 1), seed=80 + B)
    pr = dict(pr, u_i=pr["u_i"][:, :0], P=pr["P"][:M])
    args = oracle_args(pr)
    _, _, t_ref = oracle.train_loss(desc, w, *args, want_t=True)
    _, _, g_ref = oracle.train_grad(desc, w, *args, t_fixed=t_ref)
    with kns.Context(0) as ctx:
        _, g = kns.train.step(ctx, desc, torch.from_numpy(w).cuda(), gpu_batch(kns, pr, t_fixed=t_ref))
        torch.cuda.synchronize()
    # the bounds of the suite's small batches: single records' FP32 differences do not average out
    if np.abs(g_ref).max() > 0:
        assert_grad_close(g.cpu().numpy().astype(np.float64), g_ref, rtol=2e-2, frac=0.99, norm_tol=1e-2)
