"""Photon scans of any length: across the photons of an integrand block, beyond one launch's grid, and under
a workspace limit, with the bits of shorter scans of the same photons."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _scan(swf, n, L, count, n_steps=2, seed=0):
    rng = np.random.default_rng(seed)
    P = 2 * np.pi / L
    inst = swf.make_instance(swf.FIELD_PULSE_GAUSS, (1.0, 0.5, 10.0, 8.0, 0.0), (n[0], n[1], 1), (L, L, 1.0), -0.2, 0.2,
                             n_steps, p=(0.5, -1.0, 0.0), s=1, q=(-0.5, -1.0, 0.0), r=1, k=(0.0, -P, 0.0), eps=(1.0, 0.0, 0.0))
    m = rng.integers(-n[0], n[0] + 1, size=(count, 2))
    m[:, 1] = np.where(m[:, 1] == 0, 1, m[:, 1])
    k = np.concatenate([P * m, np.zeros((count, 1))], axis=1)
    return inst, k, rng.normal(size=(count, 3)), rng.normal(size=count) + 1j * rng.normal(size=count)


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("count", [1, 3, 4, 5, 7, 8, 9, 16, 17])
def test_scan_gives_each_photon_its_own_bits(prec, count):
    """Blocks of the integrand take 4 or 8 photons: full, partial and single ones, against scans of one."""
    from paper_2512_16889_gb300 import build, swf
    build.build()
    p = swf.C64 if prec == "c64" else swf.C128
    inst, k, eps, w = _scan(swf, (24, 20), 12.0, count, n_steps=5, seed=count)
    ctx = swf.Context(0)
    amps, packet = ctx.bw_photons(inst, k, eps, p, weights=w)
    for j in range(count):
        one, _ = ctx.bw_photons(inst, k[j:j + 1], eps[j:j + 1], p)
        assert np.array_equal(one[0], amps[j])
    assert np.all(np.abs(packet - w @ amps) <= 2.0**-52 * count * (np.abs(w) @ np.abs(amps)))
    ctx.close()


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("count", [32767, 32768, 65536])
def test_scan_beyond_one_launch(prec, count):
    """Two direct transforms a photon: 65535 blocks of a grid's second axis end at 32767 photons."""
    from paper_2512_16889_gb300 import build, swf
    build.build()
    p = swf.C64 if prec == "c64" else swf.C128
    inst, k, eps, w = _scan(swf, (8, 6), 6.0, count)
    ctx = swf.Context(0)
    amps, packet = ctx.bw_photons(inst, k, eps, p, weights=w)
    for a, b in ((0, 40), (count // 2 - 20, count // 2 + 21), (32740, 32767), (count - 33, count)):
        part, _ = ctx.bw_photons(inst, k[a:b], eps[a:b], p)
        assert np.array_equal(part, amps[a:b])
    assert np.all(np.abs(packet - w @ amps) <= 2.0**-52 * count * (np.abs(w) @ np.abs(amps)))
    ctx.close()


# the buffers of such a scan without scratch that grows with the photons (its sums' parts would take 16 MB
# more), and 8 KB for tables per row and field
@pytest.mark.parametrize("prec,need", [("c64", 114_003_000), ("c128", 189_813_000)])
def test_scan_under_a_workspace_limit(prec, need):
    """2000 photons and their packet on 320 x 320 with room for no more than their own buffers: the same
    bits, and again from the buffers that a scan without a limit has left."""
    from paper_2512_16889_gb300 import build, swf
    build.build()
    p = swf.C64 if prec == "c64" else swf.C128
    inst, k, eps, w = _scan(swf, (320, 320), 16 * np.pi, 2000)
    free, tight = swf.Context(0), swf.Context(0)
    tight.set_workspace_limit(need + 8192)
    a, pa = free.bw_photons(inst, k, eps, p, weights=w)
    b, pb = tight.bw_photons(inst, k, eps, p, weights=w)
    free.set_workspace_limit(1)
    c, pc = free.bw_photons(inst, k, eps, p, weights=w)
    for x, y in ((a, b), (pa, pb), (a, c), (pa, pc)):
        assert np.array_equal(x, y, equal_nan=True)  # a wrapped mode pair on the energy shell divides by zero
    free.close()
    tight.close()
