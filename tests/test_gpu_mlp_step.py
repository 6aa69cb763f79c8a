"""The training step's kernels at the edges of their ranges: rows that do not fill a
block of 8 or a stage of 32, one and several batch slices, band counts that
are no multiple of 4 or 16, hidden layers of one and of several chunks.  The
tolerance is the gradient tests' own: 2e-4 of the largest magnitude."""
import numpy as np
import pytest

from oracle import mlp_oracle as P
from tests.test_gpu_mlp import _close, _problem, melt  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,Hd", [(1, 64), (13, 192), (30, 128), (80, 256), (128, 256), (100, 320), (128, 1024)])
@pytest.mark.parametrize("B", [1, 8, 9, 33, 700, 2500])
def test_gradients_and_loss(melt, M, Hd, B):  # noqa: F811
    import torch
    x, tgt, params, mu, sd = _problem(n=3000, M=M, Hd=Hd, seed=M + Hd)
    rows = np.random.default_rng(B).integers(0, 3000, B).astype(np.int64)
    h = melt.melt_mlp_create(M, Hd, melt.pack_mlp_params(*params), mu, sd)
    grads = torch.full((melt.melt_mlp_num_params(M, Hd),), float("nan"), device="cuda")
    loss = torch.ones(1, device="cuda")
    melt.melt_mlp_grad(h, torch.from_numpy(x).cuda(), torch.from_numpy(tgt).cuda(), torch.from_numpy(rows).cuda(), B,
                       grads, loss)
    torch.cuda.synchronize()
    melt.melt_mlp_destroy(h)
    p64 = [np.asarray(p, np.float64) for p in params]
    y, cache = P.forward(p64, x[rows], mu.astype(np.float64), sd.astype(np.float64))
    ref = P.backward(p64, cache, y, tgt[rows], sd.astype(np.float64))
    for name, g, r in zip(["dW1", "db1", "dW2", "db2"], melt.unpack_mlp_params(grads.cpu().numpy(), M, Hd), ref[:4]):
        _close(g, r, (name, M, Hd, B))
    assert loss.item() == pytest.approx(1.0 + float(np.sum((y - tgt[rows]) ** 2)), rel=1e-4)
