"""All-pairs scans and C-spectra where their tiles end: against the one-pair path and against one field at
a time (both FP64 with another order of the sums: 1e-10 of the largest amplitude)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _base(n, **kw):
    L = tuple(0.5 * m if m > 1 else 1.0 for m in n)
    return dict(dict(field=("sauter_gauss", (0.8, 0.6, 2.5)), n=n, L=L, t_in=-2.0, t_out=2.0, n_steps=3, p=(0, 0, 0), s=1,
                     q=(0, 0, 0), r=1, k=(0, 0, 0), eps=(0, 0, 0), flags=()), **kw)


@pytest.mark.parametrize("n,n_e,n_p,axes", [((24, 20, 1), 1, 1, (0,)), ((24, 20, 1), 33, 1, (1,)), ((24, 20, 1), 1, 33, (0,)),
                                            ((24, 20, 1), 17, 5, (0, 1)), ((20, 32, 1), 4, 34, (1,)),
                                            ((16, 12, 10), 3, 4, (0, 1, 2)), ((45, 1, 1), 5, 2, (0,))])
def test_pair_matrix_edges(n, n_e, n_p, axes):
    from paper_2512_16889_gb300 import build, swf
    build.build()
    rng = np.random.default_rng(7)
    mom = lambda: tuple(float(rng.uniform(-0.8, 0.8)) if a in axes else 0.0 for a in range(3))
    # on a line the spin is conserved: opposite spins have amplitude zero (the oracle gives 1e-17 to 5e-14)
    spin = (lambda i: 1) if n[1] * n[2] == 1 else (lambda i: 1 - 2 * (i % 2))
    els = [_base(n, p=mom(), s=spin(i)) for i in range(n_e)]
    pos = [_base(n, q=mom(), r=spin(i)) for i in range(n_p)]
    ctx = swf.Context(0)
    mat = ctx.pair_matrix([swf.from_workload(d) for d in els], [swf.from_workload(d) for d in pos], swf.C128)
    pairs = [dict(e, q=p["q"], r=p["r"], flags=("full_n",)) for e in els for p in pos]
    ref, _ = ctx.solve([swf.from_workload(d) for d in pairs], swf.SCHWINGER, swf.C128)
    for i, r in enumerate(ref):
        got = mat[i // n_p][i % n_p]
        scale = max(abs(x) for x in r.amp)
        assert scale > 0 and max(abs(a - b) for a, b in zip(got.amp, r.amp)) <= 1e-10 * scale, i
    ctx.close()


@pytest.mark.parametrize("n,count", [((24, 20, 1), 1), ((24, 20, 1), 7), ((45, 1, 1), 9), ((16, 12, 10), 3)])
def test_spectrum_fields_of_different_momenta(n, count):
    """Fields of one call share the spinors of a mode only where they carry the same momentum along the
    trivial axes."""
    import torch

    from paper_2512_16889_gb300 import build, swf
    build.build()
    N = n[0] * n[1] * n[2]
    insts = [swf.from_workload(_base(n, p=(0.2, 0.1 * (i // 3), 0.3 * (i % 3)))) for i in range(count)]
    g = torch.Generator(device="cuda").manual_seed(5)
    psi = torch.randn(count, 8 * N, dtype=torch.float64, device="cuda", generator=g)
    ctx = swf.Context(0)
    c, prob = (torch.full((count, m * N), float("nan"), dtype=torch.float64, device="cuda") for m in (4, 2))
    ctx.spectrum_dev(insts, psi, c, prob, prec=swf.C128)
    for i in range(count):
        c1, p1 = (torch.zeros(m * N, dtype=torch.float64, device="cuda") for m in (4, 2))
        ctx.spectrum_dev(insts[i:i + 1], psi[i].contiguous(), c1, p1, prec=swf.C128)
        torch.cuda.synchronize()
        assert (c[i] - c1).abs().max().item() <= 1e-10 * c1.abs().max().item()
        assert (prob[i] - p1).abs().max().item() <= 1e-10 * p1.abs().max().item()
    ctx.close()
