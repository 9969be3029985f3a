"""Training kernels of the surrogate at the edges of their row blocks and chunks: loss and gradients
against the BF16 error model of the plain FP64 network, and an Adam step against its formula."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 15, 16, 17, 63, 65, 255, 321])
def test_gradients_and_step_at_batch_edges(batch):
    import torch

    from paper_2512_16889_gb300 import build, surrogate as S, swf, workloads as W
    from tests import bf16_bounds as BB
    build.build()
    t = W.surrogate_samples(batch, seed=31)
    X = S.features(t)
    y = (-12.0 + 3.0 * np.tanh(X[:, 0] * 5 - 1.0) + 0.5 * X[:, 3] * X[:, 4]).astype(np.float32)
    norm = np.concatenate([[0.3, 0.5, 5.5, 0, 0, 0], [11.0, 5.8, 0.7, 1.7, 1.7, 1.0], [-12.0, 0.5]]).astype(np.float32)
    p0 = S.init_params(seed=3)
    p0[np.arange(p0.size) % 7 == 0] *= 0.5
    sur = swf.Surrogate(p0, norm, max_batch=batch)
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    grad = torch.full((swf.Surrogate.param_count(),), float("nan"), device="cuda")
    loss = torch.zeros(1, device="cuda")
    sur.gradients(Xd, yd, grad, loss)
    loss64, g64, sl, sg = BB.loss_grad_sigma(p0.astype(float), X.astype(float), y.astype(float), norm.astype(float))
    g = grad.cpu().numpy().astype(float)
    assert abs(loss.item() - loss64) <= BB.K * sl
    assert np.all(np.abs(g - g64) <= BB.K * sg + 1e-12), np.max(np.abs(g - g64) / (sg + 1e-300))
    # the first step uses the same gradients: p - lr m'/(sqrt(v') + eps), m' = (1 - b1) g / (1 - b1),
    # v' = (1 - b2) g^2 / (1 - b2) with the numerators' 1 - b from b rounded to FP32 (0.999 there is off
    # by 5e-5 of 1 - b2) and the corrections rounded once from FP64
    lr = np.float32(1e-3)
    f1, f2 = (float(np.float32(1) - np.float32(b)) / float(np.float32(1 - b)) for b in (0.9, 0.999))
    sur.train_step(Xd, yd, float(lr), loss)
    p1 = sur.params().astype(float)
    want = p0.astype(float) - float(lr) * (f1 * g) / (np.sqrt(f2) * np.abs(g) + 1e-8)
    # a few FP32 roundings of the update and one of the parameter
    assert np.all(np.abs(p1 - want) <= 16 * 2.0**-24 * (np.abs(p0) + lr))
    sur.close()
