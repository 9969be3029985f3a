"""The tables a right-hand side sets up in one launch (axis factors, background phases, mode momenta,
time factors) where their blocks end: against the allocation-free entry point, whose x pass computes
the time factors itself."""
import pytest

pytestmark = pytest.mark.gpu

FIELDS = [("sauter_gauss", (0.8, 0.6, 2.5)), ("pulse_gauss", (0.3, 0.7, 4.0, 3.0)), ("single_e", (0.6, 0.5, 0.3, 0.3, 0.2))]
GRIDS = [(32, 27, 1), (30, 30, 1), (20, 64, 1), (20, 72, 1), (16, 512, 1), (8, 5, 75), (32, 1, 25), (45, 1, 1)]


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("field", FIELDS, ids=[f[0] for f in FIELDS])
def test_rhs_tables(field, n):
    """Where the time factors are computed is all that differs: at most an ulp of a factor of the local
    term, so a few units of the result's rounding."""
    import torch

    from paper_2512_16889_gb300 import build, swf
    build.build()
    inst = swf.from_workload(dict(field=field, n=n, L=tuple(0.5 * m if m > 1 else 1.0 for m in n), t_in=-4.0, t_out=4.0,
                                  n_steps=8, p=(0.3, -0.2, 0.0), s=1, q=(-0.2, 0.1, 0.0), r=-1, k=(0, 0, 0),
                                  eps=(0, 0, 0), flags=()))
    ctx = swf.Context(0)
    for prec, real in ((swf.C64, torch.float32), (swf.C128, torch.float64)):
        g = torch.Generator(device="cuda").manual_seed(3)
        psi = torch.randn(8 * n[0] * n[1] * n[2], dtype=real, device="cuda", generator=g)
        a, b = torch.full_like(psi, float("nan")), torch.full_like(psi, float("nan"))
        for bg in (0, 1):
            ctx.rhs_dev(inst, 0.37, psi, a, bg=bg, prec=prec)
            swf.rhs_noalloc(inst, 0.37, psi, b, bg=bg, prec=prec)
            torch.cuda.synchronize()
            assert (a - b).abs().max().item() <= 16 * torch.finfo(real).eps * b.abs().max().item()
    ctx.close()
