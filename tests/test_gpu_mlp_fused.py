"""The one-launch gradient of the cost model (widths 32, 64 and 128, at most 64
features) against the FP64 oracle: ragged chunks of 16 samples, fewer samples
than the cluster has blocks, one cluster and several, odd feature counts."""
import numpy as np
import pytest
import torch

import oracle
from paper_1904_10119_gb300 import fft3
from tests.test_gpu_mlp import _split

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F,H,B", [(32, 64, 128), (32, 64, 1), (31, 64, 17), (1, 32, 512), (64, 64, 513), (33, 32, 4100),
                                   (32, 128, 700), (7, 128, 40)])
def test_gradient_matches_fp64_oracle_and_repeats(F, H, B):
    m = fft3.Mlp(F, H, seed=1)
    rng = np.random.default_rng(B)
    p = rng.normal(0, 0.2, m.num_params).astype(np.float32)
    m.set_params(p)
    X = rng.normal(size=(B, F)).astype(np.float32)
    y = rng.normal(size=B).astype(np.float32)
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    grads, losses = [], []
    for _ in range(2):
        g = torch.full((p.size,), float("nan"), device="cuda")
        loss = torch.full((1,), float("nan"), device="cuda")
        assert fft3.load().fft3_mlp_grad(m.handle, Xd.data_ptr(), yd.data_ptr(), B, g.data_ptr(), loss.data_ptr(), None) == 0
        torch.cuda.synchronize()
        grads.append(g)
        losses.append(loss)
    assert torch.equal(grads[0], grads[1]) and torch.equal(losses[0], losses[1])  # sums in a fixed order
    pred, cache = oracle.mlp_forward(_split(p, F, H), X)
    ref = np.concatenate([r.ravel() for r in oracle.mlp_backward(_split(p, F, H), cache, pred, y)])
    # sums of up to H products per unit in three layers, then of B samples, each rounded to
    # 2^-24: a few units of the last place of the result's norm
    got = grads[0].cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 2e-6 * np.linalg.norm(ref)
    assert abs(losses[0].item() - oracle.mse_loss(pred, y)) <= 2e-6 * oracle.mse_loss(pred, y)
    m.close()


def test_training_keeps_no_activations():
    """The one-launch gradient needs no activations: training leaves none with the handle."""
    n, F = 1 << 18, 8
    rng = np.random.default_rng(0)
    X, y = rng.normal(size=(n, F)).astype(np.float32), rng.normal(size=n).astype(np.float32)
    m = fft3.Mlp(F, 64, seed=1)
    m.train(X[:256], y[:256], epochs=1, batch=128, lr=1e-3, seed=1)  # loads the kernels
    free = torch.cuda.mem_get_info()[0]
    m.train(X, y, epochs=1, batch=n, lr=1e-3, seed=1)
    assert free - torch.cuda.mem_get_info()[0] < 64 << 20  # activations of all samples: 6 x 64 MiB
    m.close()
