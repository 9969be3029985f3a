"""Breit-Wheeler amplitudes of photons whose mode number exceeds the grid's on an axis: the V mode is the U
mode minus the photon's, several boxes round, in both forms of the amplitude."""
import numpy as np
import pytest

from oracle import swf_oracle as O

pytestmark = pytest.mark.gpu


# photon modes per axis against grids of 16 x 12 and 15 x 18 points
@pytest.mark.parametrize("n,modes", [((16, 12, 1), (-17, 25)), ((16, 12, 1), (33, -12)), ((15, 18, 1), (-40, 18))])
@pytest.mark.parametrize("partial", [True, False])
def test_photon_modes_beyond_the_grid(n, modes, partial):
    """complex128 marches the oracle's scheme and steps: 1e-10 of |M|, as every Breit-Wheeler test."""
    from paper_2512_16889_gb300 import build, swf
    build.build()
    L = (8 * np.pi, 8 * np.pi, 1.0)
    k = (modes[0] / 4.0, modes[1] / 4.0, 0.0)
    par = np.cross(k, (0.0, 0.0, 1.0))
    eps = tuple(par / np.linalg.norm(par))
    c = dict(t_in=-3.0, t_out=3.0, n_steps=100, p=(0.25, -1.0, 0.0), q=(-0.25, -0.5, 0.0))
    ref = O.bw_amplitude(O.Field("sauter_gauss", (1.0, 0.7, 2.0)), O.Grid(n, L), c["p"], 1, c["q"], -1, O.Photon(k, eps),
                         c["t_in"], c["t_out"], c["n_steps"], form=2 if partial else 1)
    inst = swf.make_instance(swf.FIELD_SAUTER_GAUSS, (1.0, 0.7, 2.0), n, L, c["t_in"], c["t_out"], c["n_steps"], p=c["p"],
                             s=1, q=c["q"], r=-1, k=k, eps=eps, flags=swf.BW_PARTIAL if partial else 0)
    ctx = swf.Context(0)
    res, _ = ctx.solve([inst], swf.BREIT_WHEELER, swf.C128)
    got = [complex(res[0].amp[2 * j], res[0].amp[2 * j + 1]) for j in range(4)]
    scale = max(abs(t) for t in ref["terms"])
    for j in range(3):
        assert abs(got[j] - ref["terms"][j]) <= 1e-10 * scale, (j, got[j], ref["terms"][j])
    assert abs(got[3] - ref["M"]) <= 1e-10 * scale
    ctx.close()
