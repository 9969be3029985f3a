"""Grids with x as the only non-trivial axis: right-hand side and a short march against the oracle at lengths
on both sides of the rule for the radices, and each field with the same bits alone and among others."""
import numpy as np
import pytest

from oracle import swf_oracle as O
from tests.test_gpu_line_passes import FIELD, _case, _from_gpu, _to_gpu, env  # noqa: F401

pytestmark = pytest.mark.gpu

# shorter than a block and longer; 375 to 512: whole-line radices in complex128 where 16 divides the length
LENGTHS = [2, 3, 30, 45, 128, 243, 256, 270, 375, 384, 400, 405, 432, 450, 480, 486, 500, 512]


@pytest.mark.parametrize("nx", LENGTHS)
def test_right_hand_side_and_march(env, nx):  # noqa: F811
    torch, swf, ctx = env
    n = (nx, 1, 1)
    d = _case(n, 3)
    grid, fld = O.Grid(n, d["L"]), O.Field(*FIELD)
    rng = np.random.default_rng(nx)
    psi = rng.normal(size=(4,) + n) + 1j * rng.normal(size=(4,) + n)
    for bg in (0, 1):
        back = O.Background("U", d["p"], d["s"]) if bg == 0 else O.Background("V", d["q"], d["r"])
        for prec, real, eps in ((swf.C64, torch.float32, 2.0**-24), (swf.C128, torch.float64, 2.0**-53)):
            x = _to_gpu(torch, psi, real)
            out = torch.zeros_like(x)
            ctx.rhs_dev(swf.from_workload(d), 0.17, x, out, bg=bg, prec=prec)
            ref = O.rhs(fld, grid, back, O.h0_field(grid, back.offset()), 0.17, _from_gpu(x, n))
            # each butterfly level of the two transforms adds at most 4 eps, tables and pointwise work 20
            assert np.linalg.norm(_from_gpu(out, n) - ref) <= (8 * np.log2(nx) + 20) * eps * np.linalg.norm(ref), (bg, prec)
    ref = O.march_scattered(fld, grid, O.Background("U", d["p"], d["s"]), d["t_in"], d["t_out"], 3)
    for prec, real, tol in ((swf.C64, torch.float32, 2e-5), (swf.C128, torch.float64, 1e-10)):
        out = torch.zeros(8 * nx, dtype=real, device="cuda")
        ctx.march_dev([swf.from_workload(d)], out, prec=prec)
        assert np.linalg.norm(_from_gpu(out, n) - ref) <= tol * np.linalg.norm(ref), prec


@pytest.mark.parametrize("nx", [45, 128, 384, 512])
@pytest.mark.parametrize("flags", [(), ("adaptive",)])
def test_same_bits_alone_and_among_others(env, nx, flags):  # noqa: F811
    """Every field kind's component of V (A_0 and A_1) among 40 fields; controlled marches one at a time, as
    their step is shared."""
    torch, swf, ctx = env
    ds = []
    for j in range(40):
        field = (("sauter_gauss", (0.8, 0.6, 2.5)), ("single_e", (0.6, 0.5, 0.3, 0.3, 0.2)), FIELD, ("zero", ()))[j % 4]
        ds.append(dict(_case((nx, 1, 1), 6), field=field, p=(0.05 * j, -0.2, 0.1), flags=flags))
    insts = [swf.from_workload(d) for d in ds]
    for prec, real in ((swf.C64, torch.float32), (swf.C128, torch.float64)):
        alone = torch.zeros(40, 8 * nx, dtype=real, device="cuda")
        for j, inst in enumerate(insts):
            ctx.march_dev([inst], alone[j], prec=prec)
        for tune in (True, False):
            other = swf.Context(0)
            other.set_autotune(tune)
            group = torch.zeros(40, 8 * nx, dtype=real, device="cuda")
            if flags:
                for j, inst in enumerate(insts):
                    other.march_dev([inst], group[j], prec=prec)
            else:
                other.march_dev(insts, group, prec=prec)
            assert torch.equal(alone, group), prec
            other.close()
