"""y passes of long small-radix lines, whose tiles of several columns give a thread several butterflies: the
timed shapes against the fixed rule's, bit for bit, and against the other precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# lengths without register lines (243, 405, 486) in complex64; long FP64 lines; a ragged number of columns
CASES = [("c64", (486, 486, 1), 1), ("c64", (243, 243, 1), 2), ("c64", (405, 405, 1), 1), ("c64", (36, 243, 1), 3),
         ("c64", (27, 9, 243), 1), ("c128", (512, 512, 1), 1), ("c128", (45, 243, 1), 4), ("c128", (30, 480, 1), 3),
         ("c128", (2, 512, 1), 2), ("c128", (6, 5, 384), 1)]


@pytest.mark.parametrize("prec,n,count", CASES)
def test_timed_shapes_give_the_bits_of_the_fixed_rule(prec, n, count):
    import torch

    from paper_2512_16889_gb300 import build, swf
    build.build()
    L = tuple(0.3 * v if v > 1 else 1.0 for v in n)
    insts = []
    for j in range(count):
        p = tuple((0.3 + 0.1 * j, -0.2, 0.1)[a] if n[a] > 1 else 0.0 for a in range(3))
        insts.append(swf.make_instance(swf.FIELD_SAUTER_GAUSS, (0.4, 0.6, 3.0), n, L, -0.15, 0.15, 5, p=p, s=1,
                                       q=tuple(-v for v in p), r=1))
    out = {}
    for pr, real in ((swf.C64, torch.float32), (swf.C128, torch.float64)):
        for tune in (True, False):
            ctx = swf.Context(0)
            ctx.set_march_path(1)
            ctx.set_autotune(tune)
            out[pr, tune] = torch.zeros(count, 8 * int(np.prod(n)), dtype=real, device="cuda")
            ctx.march_dev(insts, out[pr, tune], prec=pr)
            ctx.close()
    p = swf.C64 if prec == "c64" else swf.C128
    assert torch.equal(out[p, True], out[p, False])
    a, b = out[swf.C64, True].double(), out[swf.C128, True]
    assert torch.linalg.norm(a - b) <= 2e-5 * torch.linalg.norm(b)
