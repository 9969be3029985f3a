"""The surrogate's inference kernel where its work is divided: one and two tiles per CTA, the second
group's first and last tile, and ragged ends, against the oracle and against itself in another order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_cta,extra", [(0, 2), (0, 129), (1, 0), (1, 1), (2, 0), (2, 1), (3, 77)])
def test_tiles_per_cta(per_cta, extra):
    """Rows are independent: a row's outputs are the same bits wherever it lies in the batch (its tile,
    group and lane), and the rows at the edges of the tiles match the FP64 network within the error
    model's 6 standard deviations."""
    import torch

    from paper_2512_16889_gb300 import build, surrogate as S, swf, workloads as W
    from tests import bf16_bounds as BB
    build.build()
    rows = per_cta * 128 * torch.cuda.get_device_properties(0).multi_processor_count + extra
    base = S.features(W.surrogate_samples(1000, seed=17)).astype(np.float32)
    norm = np.concatenate([[0.3, 0.5, 5.5, 0, 0, 0], [11.0, 5.8, 0.7, 1.7, 1.7, 1.0], [-12.0, 0.5]]).astype(np.float32)
    p0 = S.init_params(seed=3)
    p0[np.arange(p0.size) % 7 == 0] *= 0.5
    sur = swf.Surrogate(p0, norm, max_batch=64)
    x = torch.from_numpy(base).cuda().repeat(rows // 1000 + 1, 1)[:rows].contiguous()
    out = torch.full((rows + 1, 2), float("nan"), device="cuda")  # one row more than it may write
    sur.forward(x, out[:rows])
    back = torch.full((rows, 2), float("nan"), device="cuda")
    sur.forward(x.flip(0).contiguous(), back)
    sur.status()
    assert torch.isnan(out[rows]).all()
    assert torch.equal(out[:rows], back.flip(0))
    edge = sorted({r for t in (0, rows // 128 // 2, rows // 128 - 1, rows // 128) for r in (128 * t, 128 * t + 127)
                   if 0 <= r < rows} | {rows - 1})
    mu, lv, smu, slv = BB.head_sigma(p0.astype(float), x[edge].cpu().numpy().astype(float), norm.astype(float))
    got = out[edge].cpu().numpy().astype(float)
    assert np.all(np.abs(got[:, 0] - mu) <= BB.K * smu)
    assert np.all(np.abs(got[:, 1] - lv) <= BB.K * slv)
    sur.close()
