"""Calls under swf_set_workspace_limit that have room for their own buffers and no more."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _instance(swf, n, flags=0, steps=2, j=0):
    L = tuple(0.3125 * v for v in n)
    p = (0.3 + 0.01 * j, -0.2 if n[1] > 1 else 0.0, 0.0)
    return swf.make_instance(swf.FIELD_SAUTER_GAUSS, (0.3, 0.5, 5.0), n, L, -0.2, 0.2, steps, p=p, s=1,
                             q=tuple(-v for v in p), r=1, flags=flags)


def _smallest_limit(swf, call):
    """The smallest workspace limit (within 1024 bytes) at which call(context) succeeds on a fresh context."""
    def fits(limit):
        ctx = swf.Context(0)
        ctx.set_autotune(False)
        ctx.set_workspace_limit(limit)
        try:
            call(ctx)
            return True
        except swf.SwfError as e:
            assert e.status == swf.SWF_ENOMEM
            return False
        finally:
            ctx.close()
    lo, hi = 0, 1 << 16
    while not fits(hi):
        lo, hi = hi, 4 * hi
    while hi - lo > 1024:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fits(mid) else (mid, hi)
    return hi


def test_pair_number_beside_buffers_of_other_calls():
    """A context that has solved eight 256 x 256 fields on the fused kernel holds waves large enough for U
    and V of a 128 x 128 pair together, but not the pass kernels' stage buffers: with room for one wave's
    (10 arrays of 0.5 MB, the FP64 transforms of 1 MB each) U and V go one after the other."""
    from paper_2512_16889_gb300 import build, swf
    build.build()
    large = [_instance(swf, (256, 256, 1), j=j) for j in range(8)]
    pair = [_instance(swf, (128, 128, 1), flags=swf.WANT_FULL_N)]

    def first(ctx):
        ctx.solve(large, swf.SCHWINGER, swf.C64)

    free, tight = swf.Context(0), swf.Context(0)
    first(tight)
    tight.set_workspace_limit(_smallest_limit(swf, first) + 10 * (1 << 19) + 2 * (1 << 20) + (1 << 18))
    a, _ = free.solve(pair, swf.SCHWINGER, swf.C64)
    b, _ = tight.solve(pair, swf.SCHWINGER, swf.C64)
    assert bytes(a) == bytes(b)
    free.close()
    tight.close()
