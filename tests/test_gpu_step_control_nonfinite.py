"""A step-size-controlled march in which one field's values overflow ends with SWF_ENUMERIC, wherever the
field sits among the others, and leaves the context usable."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# finite parameters whose field is infinite in the march's precision
BAD = {"c64": (1e39, 0.5, 5.0), "c128": (1e308, 0.01, 5.0)}


def _instance(swf, prm, j, flags):
    return swf.make_instance(swf.FIELD_SAUTER_GAUSS, prm, (16, 12, 1), (8.0, 6.0, 1.0), -1.0, 1.0, 8,
                             p=(0.05 * j, 0.1, 0.0), s=1, q=(-0.05 * j, -0.1, 0.0), r=1, flags=flags)


# the controller's eight warps take the fields in turn
@pytest.mark.parametrize("count,bad", [(1, 0), (2, 0), (2, 1), (9, 3), (9, 8), (17, 16)])
@pytest.mark.parametrize("prec", ["c64", "c128"])
def test_overflowing_field_stops_the_march(prec, count, bad):
    import torch

    from paper_2512_16889_gb300 import build, swf
    build.build()
    p = swf.C64 if prec == "c64" else swf.C128
    good = [_instance(swf, (0.3, 0.5, 5.0), j, swf.ADAPTIVE) for j in range(count)]
    mixed = list(good)
    mixed[bad] = _instance(swf, BAD[prec], bad, swf.ADAPTIVE)
    out = torch.zeros(count * 8 * 192, dtype=torch.float32 if prec == "c64" else torch.float64, device="cuda")
    ctx = swf.Context(0)
    with pytest.raises(swf.SwfError) as ei:
        ctx.march_dev(mixed, out, prec=p)
    assert ei.value.status == swf.SWF_ENUMERIC
    ctx.march_dev(good, out, prec=p)
    again = out.cpu().numpy()
    ctx.close()
    fresh = swf.Context(0)
    fresh.march_dev(good, out, prec=p)
    assert np.all(np.isfinite(again)) and np.array_equal(again, out.cpu().numpy())
    fresh.close()


def test_overflowing_field_stops_the_breit_wheeler_march():
    from paper_2512_16889_gb300 import build, swf
    build.build()
    ctx = swf.Context(0)
    L = 8 * np.pi
    insts = [swf.make_instance(swf.FIELD_SAUTER_GAUSS, prm, (16, 16, 1), (L, L, 1.0), -1.0, 1.0, 8, p=(0.25, -1.0, 0.0),
                               s=1, q=(-0.25, -1.0, 0.0), r=1, k=(0.0, -2.0, 0.0), eps=(-1.0, 0.0, 0.0),
                               flags=swf.ADAPTIVE) for prm in ((0.3, 0.5, 5.0), BAD["c64"])]
    with pytest.raises(swf.SwfError) as ei:
        ctx.solve(insts, swf.BREIT_WHEELER, swf.C64)
    assert ei.value.status == swf.SWF_ENUMERIC
    ctx.close()
