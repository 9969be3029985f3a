"""The roundings of the training step that a compiler could contract in several ways: the loss and its
derivative with respect to the output layer's biases, and Adam's update, bit for bit in FP32."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

F = np.float32


def _fma(a, b, c):
    """a b + c in one rounding: the product of two FP32 numbers is exact in FP64, and the sum's rounding
    there decides the FP32 one (up to ties that need 29 equal bits)."""
    return (a.astype(np.float64) * np.float64(b) + np.float64(c)).astype(F)


@pytest.mark.parametrize("log_var", [0.37, -1.9])
@pytest.mark.parametrize("batch", [1, 37, 600])
def test_loss_and_bias_gradients_share_one_rounded_square(batch, log_var):
    """With zero output weights the heads are the output biases (mu, l).  A row with residual -1 gives
    w = e^{-l} as the kernel rounds it; the loss and the two bias gradients of other rows then follow from
    t = (r r) w, rounded twice: loss (t + l) / 2 (256 strided sums, then halves), dl (1 - t) / 2, dmu -r w."""
    import torch

    from paper_2512_16889_gb300 import build, surrogate as S, swf
    build.build()
    mu, l = F(0.8125), F(log_var)
    p = S.init_params(seed=9)
    p[-514:-2] = 0
    p[-2:] = mu, l
    norm = np.concatenate([np.zeros(6), np.ones(6), [0.0, 1.0]]).astype(F)
    sur = swf.Surrogate(p, norm, max_batch=batch)
    rng = np.random.default_rng(4)
    grad = torch.zeros(swf.Surrogate.param_count(), device="cuda")
    loss = torch.zeros(1, device="cuda")

    def call(y):
        x = torch.from_numpy(rng.normal(size=(len(y), 6)).astype(F)).cuda()
        sur.gradients(x, torch.from_numpy(y).cuda(), grad, loss)
        return F(loss.item()), grad[-2:].cpu().numpy()

    w = call(np.array([mu - F(1)], F))[1][0]
    for _ in range(200 if batch == 1 else 4):
        y = rng.normal(scale=1.5, size=batch).astype(F)
        r = y - mu
        t = (r * r) * w
        part = np.zeros(256, F)
        dmu = dl = F(0)
        for b in range(batch):
            part[b % 256] += F(0.5) * (t[b] + l)
            dmu += (-r[b] * w) / F(batch)
            dl += (F(0.5) * (F(1) - t[b])) / F(batch)
        half = 128
        while half:
            part[:half] += part[half:2 * half]
            half //= 2
        got, g = call(y)
        assert got == part[0] / F(batch)
        assert g[0] == dmu and g[1] == dl
    sur.close()


def test_adam_update_bits():
    """m' = (1 - b1) g + (b1 m), v' = ((1 - b2) g) g + (b2 v), each product beside the plus sign in one
    rounding with it; p - (lr (m'/c1)) / (sqrt(v'/c2) + eps), every operation rounded."""
    import torch

    from paper_2512_16889_gb300 import build, surrogate as S, swf, workloads as W
    build.build()
    t = W.surrogate_samples(128, seed=17)
    X = S.features(t)
    y = (-10.0 + 2.0 * np.tanh(X[:, 0] * 4) + 0.3 * X[:, 4]).astype(F)
    p = S.init_params(seed=2)
    sur = swf.Surrogate(p, S.normalisation(X, y), max_batch=128)
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    grad = torch.zeros(swf.Surrogate.param_count(), device="cuda")
    loss = torch.zeros(1, device="cuda")
    lr, b1, b2, eps = F(1e-3), F(0.9), F(0.999), F(1e-8)
    m, v = np.zeros_like(p), np.zeros_like(p)
    for k in range(1, 4):
        sur.gradients(Xd, yd, grad, loss)
        g = grad.cpu().numpy()
        m = _fma(g, F(1) - b1, b1 * m)
        v = _fma((F(1) - b2) * g, g, b2 * v)
        c1, c2 = F(1 - 0.9**k), F(1 - 0.999**k)
        p = p - (lr * (m / c1)) / (np.sqrt(v / c2) + eps)
        sur.train_step(Xd, yd, float(lr), loss)
        assert np.array_equal(sur.params(), p)
    sur.close()
