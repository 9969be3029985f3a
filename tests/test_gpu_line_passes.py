"""The pass kernels of the march at every length that has kernels of its own and at the edges of the
others (lengths 1 to 5, 3^5 and 2 3^5, trivial x or y axes): right-hand side and a short march against
the oracle, and grouped against single-group marches."""
import os
import re

import numpy as np
import pytest

from oracle import swf_oracle as O

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
with open(os.path.join(ROOT, "paper_2512_16889_gb300", "csrc", "swf_line_list.h")) as _f:
    LENGTHS = sorted({int(m) for m in re.findall(r"X\((\d+),", _f.read())})
# partners for the other axis: neither multiples of the column tile nor with kernels of their own
PARTNERS = (9, 10, 15, 12)
EDGES = [(1, 48, 1), (1, 20, 32), (32, 1, 45), (5, 8, 1), (2, 64, 1), (3, 486, 1), (486, 3, 1), (243, 4, 1), (40, 36, 32),
         (27, 20, 50), (1, 3, 6)]
GRIDS = [(n, PARTNERS[i % 4], 1) for i, n in enumerate(LENGTHS)] + [(PARTNERS[i % 4], n, 1) for i, n in enumerate(LENGTHS)] + EDGES
FIELD = ("pulse_gauss", (0.8, 0.9, 4.0, 3.0, 0.0))  # its time factor depends on y


@pytest.fixture(scope="module")
def env():
    import torch

    from paper_2512_16889_gb300 import swf
    ctx = swf.Context(0)
    yield torch, swf, ctx
    ctx.close()


def _case(n, steps):
    L = tuple(0.4 * v if v > 1 else 1.0 for v in n)
    h = 0.25 * 0.4
    return dict(field=FIELD, n=n, L=L, t_in=-0.5 * steps * h, t_out=0.5 * steps * h, n_steps=steps, p=(0.3, -0.2, 0.1),
                s=1, q=(-0.3, 0.2, -0.1), r=-1, k=(0, 0, 0), eps=(0, 0, 0), flags=())


def _to_gpu(torch, psi, real):
    v = np.ascontiguousarray(np.transpose(psi, (0, 3, 2, 1)))  # [4][nz][ny][nx]
    return torch.from_numpy(np.stack([v.real, v.imag], axis=-1)).to(real).cuda().contiguous()


def _from_gpu(t, n):
    v = t.double().cpu().numpy().reshape(4, n[2], n[1], n[0], 2)
    return np.transpose(v[..., 0] + 1j * v[..., 1], (0, 3, 2, 1))


@pytest.mark.parametrize("n", GRIDS, ids=lambda n: "x".join(map(str, n)))
def test_right_hand_side_and_march_at_every_length(env, n):
    torch, swf, ctx = env
    d = _case(n, 3)
    grid, fld = O.Grid(n, d["L"]), O.Field(*FIELD)
    rng = np.random.default_rng(n[0] * 1000 + n[1])
    psi = rng.normal(size=(4,) + n) + 1j * rng.normal(size=(4,) + n)
    levels = np.log2(np.prod(n))
    for bg in (0, 1):
        back = O.Background("U", d["p"], d["s"]) if bg == 0 else O.Background("V", d["q"], d["r"])
        for prec, real, eps in ((swf.C64, torch.float32, 2.0**-24), (swf.C128, torch.float64, 2.0**-53)):
            x = _to_gpu(torch, psi, real)
            out = torch.zeros_like(x)
            ctx.rhs_dev(swf.from_workload(d), 0.17, x, out, bg=bg, prec=prec)
            ref = O.rhs(fld, grid, back, O.h0_field(grid, back.offset()), 0.17, _from_gpu(x, n))
            got = _from_gpu(out, n)
            # each butterfly level of the two transforms adds at most 4 eps, tables and pointwise work 20
            assert np.linalg.norm(got - ref) <= (8 * levels + 20) * eps * np.linalg.norm(ref), (bg, prec)
    ref = O.march_scattered(fld, grid, O.Background("U", d["p"], d["s"]), d["t_in"], d["t_out"], 3)
    for prec, real, tol in ((swf.C64, torch.float32, 2e-5), (swf.C128, torch.float64, 1e-10)):
        out = torch.zeros(4 * int(np.prod(n)) * 2, dtype=real, device="cuda")
        ctx.march_dev([swf.from_workload(d)], out, prec=prec)
        assert np.linalg.norm(_from_gpu(out, n) - ref) <= tol * np.linalg.norm(ref), prec


def test_grouped_marches_of_line_lengths_equal_single_group_marches(env):
    torch, swf, _ = env
    ds = []
    for n in ((64, 48, 1), (96, 36, 1), (27, 80, 1)):
        for px in (-0.3, 0.4):
            ds.append(dict(_case(n, 5), p=(px, 0.1, 0.0), q=(-px, 0.0, 0.0), flags=("spectrum", "full_n")))
    for prec in (swf.C64, swf.C128):
        got = []
        for mode in (2, 0):
            ctx = swf.Context(0)
            ctx.set_multi_grid(mode)
            res, spec = ctx.solve([swf.from_workload(dict(d, t_in=-0.25, t_out=0.25)) for d in ds], swf.SCHWINGER, prec)
            got.append((np.frombuffer(res, dtype=np.float64).copy(), spec))
            ctx.close()
        assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
        assert np.all(np.isfinite(got[0][0]))
