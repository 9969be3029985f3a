"""The full pair number with the U and V fields in one march (small groups) against one march after the
other (a workspace limit keeps them apart): the same bits, and the same answers under a limit."""
import pytest

pytestmark = pytest.mark.gpu

GROUPS = [("sauter_gauss", (0.8, 0.6, 2.5), (32, 24, 1), 1), ("single_e", (0.6, 0.5, 0.3, 0.3, 0.2), (16, 12, 10), 3),
          ("sauter_gauss", (0.8, 0.6, 2.5), (45, 1, 1), 2), ("pulse_gauss", (0.5, 0.7, 3.0, 3.0, 0.0), (27, 1, 20), 2),
          ("double_e", (0.4, 0.5, 0.3, 0.3, 0.2, 1.0), (256, 128, 1), 7), ("sauter_gauss", (0.8, 0.6, 2.5), (256, 128, 1), 8)]


def _instances(swf, field, prm, n, count):
    L = tuple(0.5 * m if m > 1 else 1.0 for m in n)
    out = []
    for i in range(count):
        p = tuple(6.283185307179586 * (i // 2 + 1 + a) / L[a] if n[a] > 1 else 0.0 for a in range(3))
        out.append(swf.from_workload(dict(field=(field, prm), n=n, L=L, t_in=-2.0, t_out=2.0, n_steps=5, p=p, s=1 - 2 * (i % 2),
                                          q=tuple(-x for x in p), r=1, k=(0, 0, 0), eps=(0, 0, 0),
                                          flags=("full_n", "spectrum"))))
    return out


def _values(res):
    return [tuple(r.amp) + tuple(r.prob) + tuple(r.diag) for r in res]


@pytest.mark.parametrize("field,prm,n,count", GROUPS, ids=lambda v: str(v) if isinstance(v, (str, int)) else None)
@pytest.mark.parametrize("prec", ["c64", "c128"])
def test_pair_march_same_bits(field, prm, n, count, prec):
    """Groups of every dimension, odd lengths, both spins of a momentum (marched once), and the sizes on
    either side of the line."""
    import numpy as np

    from paper_2512_16889_gb300 import build, swf
    build.build()
    p = swf.C64 if prec == "c64" else swf.C128
    insts = _instances(swf, field, prm, n, count)
    together, apart = swf.Context(0), swf.Context(0)
    apart.set_workspace_limit(1 << 40)
    ra, sa = together.solve(insts, swf.SCHWINGER, p)
    rb, sb = apart.solve(insts, swf.SCHWINGER, p)
    assert _values(ra) == _values(rb)
    assert np.array_equal(sa, sb)
    assert together.fields_marched() == apart.fields_marched()
    # a limit below what the context holds: the same call is answered from the buffers it has
    together.set_workspace_limit(1)
    rc, _ = together.solve(insts, swf.SCHWINGER, p)
    assert _values(rc) == _values(ra)
    together.close()
    apart.close()
