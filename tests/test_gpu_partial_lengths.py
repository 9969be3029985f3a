"""The partial-integration form over the lengths of its x pass: complex64 (register lines and small radices)
against the complex128 march of the same instance, which the oracle pins."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# register lines of several rows a block and one, blocks that are no multiple of 32 threads, unequal
# radices (5 x 6, 5 x 9, 6 x 8, 10 x 10, 5 x 25, 9 x 18, 15 x 18, 18 x 25, 16 x 32), then two lengths without one
@pytest.mark.parametrize("nx", [30, 45, 48, 100, 125, 162, 270, 450, 512, 27, 405])
def test_complex64_against_complex128(nx):
    """5e-5 of the larger of the term and M, the bound of every complex64 Breit-Wheeler test."""
    from paper_2512_16889_gb300 import build, swf
    build.build()
    ny, d = 9, 0.5
    L = (nx * d, ny * d, 1.0)
    k = (2 * np.pi * 3 / L[0], 2 * np.pi * 2 / L[1], 0.0)
    eps = np.array([k[1], -k[0], 0.0]) / np.hypot(k[0], k[1])
    insts = [swf.make_instance(swf.FIELD_SAUTER_GAUSS, (1.0, 0.7, 2.0), (nx, ny, 1), L, -2.0, 2.0, 40, p=(px, -0.5, 0.0),
                               s=1, q=(-0.2, 0.3, 0.0), r=r, k=k, eps=tuple(eps), flags=swf.BW_PARTIAL)
             for px, r in ((0.25, 1), (-0.4, -1), (0.1, 1))]
    ctx = swf.Context(0)
    got, ref = ([np.array(v.amp[0:8:2]) + 1j * np.array(v.amp[1:8:2]) for v in ctx.solve(insts, swf.BREIT_WHEELER, p)[0]]
                for p in (swf.C64, swf.C128))
    for a, b in zip(got, ref):
        assert np.all(np.abs(a - b) <= 5e-5 * np.maximum(np.abs(b), abs(b[3]))), (a, b)
    again = ctx.solve(insts, swf.BREIT_WHEELER, swf.C64)[0]
    assert all(np.array_equal(np.array(v.amp[0:8:2]) + 1j * np.array(v.amp[1:8:2]), a) for v, a in zip(again, got))
    ctx.close()
