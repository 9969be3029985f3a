"""The calls whose time is followed: what a program that uses the solver has it do.

Each case is one pass through a public entry point of ``paper_2512_16889_gb300.swf`` (a
``Context`` or a ``Surrogate``).  ``listed()`` names twelve of them, from the smallest call to the
largest, ``draw()`` gives more from the same ranges, ``prepare()`` makes what the program has in
hand before the call, ``run()`` is the call, ``work()`` what it cannot do without and ``exact()``
what it returns, in 64 bits, by plain torch.

Marches are shortened: a solve repeats the same step hundreds or thousands of times, so a few
steps in the middle of the pulse (where the gauge field is not zero) stand for it.

Results of a complex64 march are kept as single-precision numbers, as a program that chose that
march keeps them; those of a complex128 march and of the FP64 projections as double.
"""
import math

import numpy as np
import torch

from paper_2512_16889_gb300 import swf

FIELDS = {"sauter_gauss": swf.FIELD_SAUTER_GAUSS, "pulse_gauss": swf.FIELD_PULSE_GAUSS,
          "single_e": swf.FIELD_SINGLE_E, "double_e": swf.FIELD_DOUBLE_E}
PREC = {"c64": swf.C64, "c128": swf.C128}
REAL = {"c64": torch.float32, "c128": torch.float64}

# lengths a grid axis can have: products of 2, 3 and 5
LENGTHS = sorted(2**a * 3**b * 5**c for a in range(10) for b in range(6) for c in range(4)
                 if 16 <= 2**a * 3**b * 5**c <= 512)


def listed():
    return [
        # one right-hand side for a program's own integrator, on the smallest grid in earnest: latency
        {"name": "rhs_small", "call": "rhs", "prec": "c64", "field": "sauter_gauss", "nx": 64, "ny": 64, "nz": 1},
        # one FP64 solve as a first look at a field: full pair number and C-spectrum, 128 x 128
        {"name": "solve_fp64_single", "call": "solve", "prec": "c128", "field": "sauter_gauss", "nx": 128, "ny": 128,
         "nz": 1, "count": 1, "steps": 60, "full": True, "adaptive": False},
        # the batched momentum scan: 8 x 8 momenta, both spins, 256 x 256
        {"name": "march_batched", "call": "march", "prec": "c64", "field": "sauter_gauss", "nx": 256, "ny": 256,
         "nz": 1, "count": 128, "steps": 16, "adaptive": False},
        # a few momenta on a ragged box with the paper's step-size control
        {"name": "march_adaptive", "call": "march", "prec": "c64", "field": "double_e", "nx": 240, "ny": 135,
         "nz": 1, "count": 6, "steps": 80, "adaptive": True},
        # (3+1)D: one electron on 256^3
        {"name": "march_3d", "call": "march", "prec": "c64", "field": "sauter_gauss", "nx": 256, "ny": 256, "nz": 256,
         "count": 1, "steps": 4, "adaptive": False},
        # Breit-Wheeler pairs on uneven grids (192, 256, 320, 384)
        {"name": "bw_uneven", "call": "bw", "prec": "c64", "sizes": "192,256,320,384", "count": 32, "steps": 16,
         "partial": False},
        # the partial-integration form of the same amplitude, in FP64, a few pairs on a mid-sized grid
        {"name": "bw_partial_fp64", "call": "bw", "prec": "c128", "sizes": "160", "count": 3, "steps": 12,
         "partial": True},
        # one pair and a list of photons
        {"name": "bw_photons", "call": "photons", "prec": "c64", "nx": 192, "ny": 192, "count": 64, "steps": 50},
        # the momentum cross section of the paper's double field: 100 x 100 pairs
        {"name": "pair_matrix", "call": "pairs", "prec": "c64", "field": "double_e", "nx": 256, "ny": 128, "nz": 1,
         "electrons": 100, "positrons": 100, "steps": 12},
        # C-spectra of waves that a program has marched and kept
        {"name": "spectrum", "call": "spectrum", "prec": "c64", "nx": 256, "ny": 256, "nz": 1, "count": 16},
        # the surrogate over a parameter scan
        {"name": "surrogate_scan", "call": "forward", "rows": 1000000},
        # the surrogate's training: mini-batches of 256
        {"name": "surrogate_train", "call": "train", "batch": 256, "batches": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _length(rng, lo, hi):
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((n for n in LENGTHS if lo <= n <= hi), key=lambda n: abs(math.log(n / x)))


def _grid(rng, sites):
    """A grid of at most `sites` points: one, two or three axes, of any lengths."""
    while True:
        axes = rng.choices((1, 2, 3), (1, 7, 3))[0]
        n = [_length(rng, 32 if axes < 3 else 16, 512 if axes < 3 else 256) if a < axes else 1 for a in range(3)]
        if n[0] * n[1] * n[2] <= sites:
            return n


def _counts(rng, sites, most, most_count, most_steps):
    """(count, steps) with count * steps * sites <= most."""
    steps = _log_int(rng, 4, most_steps)
    count = _log_int(rng, 1, most_count)
    while count * steps * sites > most and count > 1:
        count = max(1, count // 2)
    while count * steps * sites > most and steps > 2:
        steps = max(2, steps // 2)
    return count, steps


def draw(rng):
    call = rng.choices(("rhs", "march", "solve", "bw", "photons", "pairs", "spectrum", "forward", "train"),
                       (2, 5, 2, 3, 1, 2, 2, 2, 2))[0]
    prec = rng.choices(("c64", "c128"), (2, 1))[0]
    field = rng.choice(("sauter_gauss", "sauter_gauss", "single_e", "double_e", "pulse_gauss"))
    work = 5e7 if prec == "c64" else 5e6  # site-updates
    if call == "rhs":
        nx, ny, nz = _grid(rng, 1 << (24 if prec == "c64" else 22))
        return {"call": call, "prec": prec, "field": field, "nx": nx, "ny": ny, "nz": nz}
    if call in ("march", "solve"):
        nx, ny, nz = _grid(rng, work / 4)
        adaptive = rng.random() < 0.25
        count, steps = _counts(rng, nx * ny * nz, work / 2, 64, 100)
        full = rng.random() < 0.5
        d = {"call": call, "prec": prec, "field": field, "nx": nx, "ny": ny, "nz": nz, "count": count, "steps": steps,
             "adaptive": adaptive}
        return dict(d, full=full) if call == "solve" else d
    if call == "bw":
        sizes = [_length(rng, 48, 400) for _ in range(rng.choice((1, 1, 2, 4)))]
        count, steps = _counts(rng, 2 * max(sizes)**2, work / 2, 32, 60)
        return {"call": call, "prec": prec, "sizes": ",".join(str(n) for n in sizes), "count": max(count, len(sizes)),
                "steps": steps, "partial": rng.random() < 0.4}
    if call == "photons":
        nx, ny = _length(rng, 48, 320), _length(rng, 48, 320)
        count, steps = _log_int(rng, 2, 100), _counts(rng, 2 * nx * ny, work / 4, 1, 100)[1]
        return {"call": call, "prec": prec, "nx": nx, "ny": ny, "count": count, "steps": steps}
    if call == "pairs":
        nx, ny = _length(rng, 48, 256), _length(rng, 32, 256)
        electrons, positrons = _log_int(rng, 2, 100), _log_int(rng, 2, 100)
        steps = max(2, min(_log_int(rng, 4, 24), int(work / 2 / ((electrons + positrons) * nx * ny))))
        return {"call": call, "prec": prec, "field": field, "nx": nx, "ny": ny, "nz": 1, "electrons": electrons,
                "positrons": positrons, "steps": steps}
    if call == "spectrum":
        nx, ny, nz = _grid(rng, 1 << 21)
        return {"call": call, "prec": prec, "nx": nx, "ny": ny, "nz": nz,
                "count": max(1, min(_log_int(rng, 1, 64), (1 << 22) // (nx * ny * nz)))}
    if call == "forward":
        return {"call": call, "rows": _log_int(rng, 1, 1000000)}
    return {"call": call, "batch": _log_int(rng, 32, 4096), "batches": _log_int(rng, 1, 8)}


# ------------------------------------------------------------------ the program's side
_ctx = None


def _context():
    """One context, kept for the life of the program."""
    global _ctx
    if _ctx is None:
        _ctx = swf.Context(0)
    return _ctx


def _box(n):
    """Box lengths: 40 for axes of 128 points and more (as the batched workload), the same spacing below."""
    return [min(40.0, 0.3125 * v) if v > 1 else 1.0 for v in n]


def _prm(kind, rng):
    """Parameters of one field kind, as a scan varies them."""
    if kind == "sauter_gauss":
        return [rng.uniform(0.15, 0.45), rng.uniform(0.2, 0.8), rng.uniform(3.0, 8.0)]
    if kind == "pulse_gauss":
        return [rng.uniform(0.5, 1.0), 0.5, 10.0, 8.0, 0.0]
    e0 = rng.uniform(0.2, 0.4)
    return [e0, e0, e0 / 2, e0 / 2, e0 / 2] + ([1.75 / (e0 / 2)] if kind == "double_e" else [])


def _dicts(case, seed):
    """The instances of a case as plain dicts (the same for prepare() and exact())."""
    rng = np.random.default_rng(seed)
    call = case["call"]
    out = []
    if call in ("bw", "photons"):
        sizes = [int(v) for v in case["sizes"].split(",")] if call == "bw" else [case["nx"]]
        box = 16.0 * math.pi
        prm = [rng.uniform(0.8, 1.2), 0.5, 10.0, 8.0, 0.0]
        h = 0.25 * box / max(sizes + [case.get("ny", 1)])
        t = 0.5 * case["steps"] * h
        for i in range(case["count"] if call == "bw" else 1):
            n = sizes[i % len(sizes)]
            P = rng.uniform(-1.5, 1.5)
            out.append(dict(field="pulse_gauss", prm=prm, n=(n, case.get("ny", n), 1), L=(box, box, 1.0), t_in=-t, t_out=t,
                            steps=case["steps"], p=(P, -1.0, 0.0), s=int(rng.choice([1, -1])), q=(-P, -1.0, 0.0),
                            r=int(rng.choice([1, -1])), k=(0.0, -2.0, 0.0), eps=(-1.0, 0.0, 0.0),
                            flags=swf.BW_PARTIAL if case.get("partial") else 0))
        return out
    n = (case["nx"], case["ny"], case["nz"])
    L = _box(n)
    steps = case.get("steps", 1)
    t = 0.5 * steps * 0.25 * min(L[a] / n[a] for a in range(3) if n[a] > 1)
    kind = case.get("field", "sauter_gauss")
    flags = (swf.ADAPTIVE if case.get("adaptive") else 0) | (swf.WANT_FULL_N if case.get("full") else 0)
    if call == "solve":
        flags |= swf.WANT_SPECTRUM
    if call == "pairs":  # one field, momenta on the grid's modes along x
        prm = _prm(kind, rng)
        base = dict(field=kind, prm=prm, n=n, L=L, t_in=-t, t_out=t, steps=steps, k=(0, 0, 0), eps=(0, 0, 0), flags=0)
        py = 2 * math.pi / L[1] * int(rng.integers(-2, 3))
        for m, is_e in ((case["electrons"], True), (case["positrons"], False)):
            for j in range(m):
                mom = (2 * math.pi / L[0] * (j - m // 2), py if is_e else -py, 0.0)
                out.append(dict(base, p=mom if is_e else (0.0, 0.0, 0.0), s=1, q=(0.0, 0.0, 0.0) if is_e else mom, r=1))
        return out
    for _ in range(case.get("count", 1)):
        p = [rng.uniform(-1, 1) if n[a] > 1 else 0.0 for a in range(3)]
        out.append(dict(field=kind, prm=_prm(kind, rng), n=n, L=L, t_in=-t, t_out=t, steps=steps, p=tuple(p),
                        s=int(rng.choice([1, -1])), q=tuple(-v for v in p), r=int(rng.choice([1, -1])), k=(0, 0, 0),
                        eps=(0, 0, 0), flags=flags))
    return out


def _instance(d):
    return swf.make_instance(FIELDS[d["field"]], d["prm"], d["n"], d["L"], d["t_in"], d["t_out"], d["steps"], p=d["p"],
                             s=d["s"], q=d["q"], r=d["r"], k=d["k"], eps=d["eps"], flags=d["flags"])


def _waves(case, seed):
    """Waves [count][4][nz][ny][nx] (re, im) of a march's smoothness: noise under a Gaussian envelope."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = (case["nx"], case["ny"], case["nz"])
    psi = torch.randn(case.get("count", 1), 4, n[2], n[1], n[0], 2, generator=g, device="cuda", dtype=REAL[case["prec"]])
    for a in range(3):
        x = (torch.arange(n[a], device="cuda", dtype=psi.dtype) - n[a] / 2) / n[a] if n[a] > 1 else torch.zeros(1, device="cuda", dtype=psi.dtype)
        psi *= torch.exp(-8 * x * x).reshape([n[a] if b == 2 - a else 1 for b in range(3)] + [1])
    return psi


def _photons(case, seed):
    """Photons k = (2 pi m / L, -2, 0), each with a polarisation transverse to it, and packet weights."""
    rng = np.random.default_rng(seed + 1)
    m = np.arange(case["count"]) // 2 - case["count"] // 4
    k = np.stack([m / 8.0, np.full(len(m), -2.0), np.zeros(len(m))], axis=1)
    par = np.stack([k[:, 1], -k[:, 0], 0 * k[:, 0]], axis=1) / np.linalg.norm(k, axis=1)[:, None]
    eps = np.where((np.arange(len(m)) % 2 == 0)[:, None], par, np.array([0.0, 0.0, -1.0]))
    w = np.exp(-(m / 8.0)**2) * np.exp(2j * math.pi * rng.uniform(size=len(m)))
    return k, eps, w


_NORM = np.array([0.3, 0.5, 5.5, 0, 0, 0, 1 / 0.0866, 1 / 0.173, 1 / 1.44, 1 / 0.577, 1 / 0.577, 1, -9.0, 1 / 3.0], np.float32)


def _weights(seed):
    """He-style weights of the 6-256-256-256-256-2 network."""
    rng = np.random.default_rng(seed)
    p = []
    for i, o in ((6, 256), (256, 256), (256, 256), (256, 256), (256, 2)):
        p += [rng.normal(scale=math.sqrt(2.0 / i) * (0.1 if o == 2 else 1.0), size=i * o), 0.1 * rng.normal(size=o)]
    return np.concatenate(p).astype(np.float32)


def _samples(rows, seed):
    """Rows (E, omega, lambda, p_x, p_y, s) of a scan and targets of the size of ln P."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand(rows, 6, generator=g, device="cuda")
    lo = torch.tensor([0.15, 0.2, 3.0, -1.0, -1.0, 0.0], device="cuda")
    hi = torch.tensor([0.45, 0.8, 8.0, 1.0, 1.0, 1.0], device="cuda")
    x = lo + (hi - lo) * u
    x[:, 5] = torch.where(u[:, 5] < 0.5, -1.0, 1.0)
    y = -math.pi / x[:, 0] + torch.log(x[:, 2]) - 2.0 * (x[:, 3]**2 + x[:, 4]**2) / x[:, 0] * x[:, 1]
    return x.contiguous(), y.contiguous()


def prepare(case, seed):
    call = case["call"]
    if call == "forward":
        sur = swf.Surrogate(_weights(seed), _NORM, max_batch=1)
        x, _ = _samples(case["rows"], seed)
        return {"call": call, "sur": sur, "x": x, "out": torch.zeros(case["rows"], 2, device="cuda")}
    if call == "train":
        sur = swf.Surrogate(_weights(seed), _NORM, max_batch=case["batch"])
        x, y = _samples(case["batch"] * case["batches"], seed)
        return {"call": call, "sur": sur, "x": x.split(case["batch"]), "y": y.split(case["batch"]),
                "loss": torch.zeros(1, device="cuda")}
    ds = _dicts(case, seed)
    s = {"call": call, "ctx": _context(), "prec": PREC[case["prec"]], "insts": [_instance(d) for d in ds],
         "single": case["prec"] == "c64"}
    sites = case.get("nx", 1) * case.get("ny", 1) * case.get("nz", 1)
    if call == "rhs":
        s["psi"] = _waves(case, seed)[0]
        s["out"] = torch.zeros_like(s["psi"])
    elif call == "march":
        s["out"] = torch.zeros(case["count"], 4, case["nz"], case["ny"], case["nx"], 2, device="cuda", dtype=REAL[case["prec"]])
    elif call == "spectrum":
        s["psi"] = _waves(case, seed)
        s["c"] = torch.zeros(case["count"], 2, sites, 2, device="cuda", dtype=torch.float64)
        s["prob"] = torch.zeros(case["count"], 2, sites, device="cuda", dtype=torch.float64)
    elif call == "photons":
        s["photons"] = _photons(case, seed)
    elif call == "pairs":
        s["electrons"], s["positrons"] = s["insts"][:case["electrons"]], s["insts"][case["electrons"]:]
    return s


def _numbers(res, single):
    """Results as arrays: complex amplitudes, probabilities, norms."""
    v = np.frombuffer(res, dtype=np.float64).reshape(-1, 12) if not isinstance(res, list) else np.stack(
        [np.frombuffer(r, dtype=np.float64) for row in res for r in row])
    amp, prob, diag = v[:, 0:8:2] + 1j * v[:, 1:8:2], v[:, 8:10], v[:, 10:12]
    if single:
        return amp.astype(np.complex64), prob.astype(np.float32), diag.astype(np.float32)
    return amp, prob.copy(), diag.copy()


def run(state):
    s, call = state, state["call"]
    if call == "forward":
        s["sur"].forward(s["x"], s["out"])
        return s["out"]
    if call == "train":
        for x, y in zip(s["x"], s["y"]):
            s["sur"].train_step(x, y, 1e-3, s["loss"])
        return {"params": s["sur"].params(), "loss": s["loss"]}
    ctx = s["ctx"]
    if call == "rhs":
        ctx.rhs_dev(s["insts"][0], 0.125, s["psi"], s["out"], prec=s["prec"])
        return s["out"]
    if call == "march":
        ctx.march_dev(s["insts"], s["out"], prec=s["prec"])
        return s["out"]
    if call == "spectrum":
        ctx.spectrum_dev(s["insts"], s["psi"], s["c"], s["prob"], prec=s["prec"])
        return {"c": s["c"], "prob": s["prob"]}
    if call == "solve":
        res, spec = ctx.solve(s["insts"], swf.SCHWINGER, s["prec"])
        amp, prob, diag = _numbers(res, s["single"])
        return {"amp": amp, "prob": prob, "diag": diag, "spectrum": spec.astype(np.float32) if s["single"] else spec}
    if call == "bw":
        amp, prob, diag = _numbers(ctx.solve(s["insts"], swf.BREIT_WHEELER, s["prec"])[0], s["single"])
        return {"amp": amp, "prob": prob, "diag": diag}
    if call == "photons":
        amps, packet = ctx.bw_photons(s["insts"][0], s["photons"][0], s["photons"][1], s["prec"], s["photons"][2])
        return {"amps": amps.astype(np.complex64), "packet": packet.astype(np.complex64)} if s["single"] else {"amps": amps, "packet": packet}
    amp, prob, diag = _numbers(ctx.pair_matrix(s["electrons"], s["positrons"], s["prec"]), s["single"])
    return {"amp": amp, "prob": prob, "diag": diag}


# ------------------------------------------------------------------ what a pass cannot do without
def _fft_flops(n):
    N = n[0] * n[1] * n[2]
    return 5.0 * N * sum(math.log2(v) for v in n if v > 1)


def _rhs_flops(n):
    """One right-hand side: forward and inverse transforms of four components, H0 (56 flops a mode)
    and the local term (48 a site)."""
    return 8.0 * _fft_flops(n) + 104.0 * n[0] * n[1] * n[2]


def work(case):
    call = case["call"]
    net = 2.0 * (6 * 256 + 3 * 256 * 256 + 2 * 256)
    if call == "forward":
        return {"bytes": 32.0 * case["rows"] + 4.0 * 199938, "flops": net * case["rows"]}
    if call == "train":  # forward and backward, and Adam's read and write of three arrays a batch
        return {"bytes": case["batches"] * (28.0 * case["batch"] + 24.0 * 199938),
                "flops": case["batches"] * 3.0 * net * case["batch"]}
    e = 8.0 if case["prec"] == "c64" else 16.0
    if call in ("bw", "photons"):
        sizes = [int(v) for v in case["sizes"].split(",")] if call == "bw" else [case["nx"]]
        total = {"bytes": 0.0, "flops": 0.0}
        for i in range(case["count"] if call == "bw" else 1):
            n = (sizes[i % len(sizes)], case.get("ny", sizes[i % len(sizes)]), 1)
            N = n[0] * n[1]
            stage = 6 * 2 * _rhs_flops(n) + 2 * 26 * 16.0 * N  # right-hand sides and stage sums of U and V
            integrand = 5 * 150.0 * N * (case["count"] if call == "photons" else 1)
            if case.get("partial"):
                integrand = 5 * (8.0 * _fft_flops(n) + 600.0 * N)
            total["flops"] += case["steps"] * (stage + integrand)
            total["bytes"] += 2 * 4 * e * N
        return total
    n = (case["nx"], case["ny"], case["nz"])
    N = n[0] * n[1] * n[2]
    if call == "rhs":
        return {"bytes": 8 * e * N, "flops": _rhs_flops(n)}
    if call == "spectrum":
        return {"bytes": case["count"] * N * (4 * e + 48.0), "flops": case["count"] * (4 * _fft_flops(n) + 100.0 * N)}
    step = 6 * _rhs_flops(n) + 26 * 16.0 * N
    fields = case["electrons"] + case["positrons"] if call == "pairs" else case["count"] * (2 if case.get("full") else 1)
    total = {"bytes": fields * 4 * e * N, "flops": fields * case["steps"] * step}
    if call == "solve":
        total["bytes"] += case["count"] * 16.0 * N
        total["flops"] += fields * 4 * _fft_flops(n)
    if call == "pairs":
        total["flops"] += fields * 4 * _fft_flops(n) + 8.0 * 4 * N * case["electrons"] * case["positrons"]
        total["bytes"] += 96.0 * case["electrons"] * case["positrons"]
    return total


# ------------------------------------------------------------------ the same, in 64 bits, by plain torch
_F64 = torch.float64
_R = {1: np.array([1, 1, 1, 1]) / 2.0, -1: np.array([1, -1, -1, 1]) / 2.0}
_SIG = [np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]], complex)]
_Z = np.zeros((2, 2), complex)
_ALPHA = [np.block([[_Z, s], [s, _Z]]) for s in _SIG]
_BETA = np.diag([1, 1, -1, -1]).astype(complex)
_DP_C = [0, 1 / 5, 3 / 10, 4 / 5, 8 / 9, 1, 1]
_DP_A = [[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9], [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
         [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656],
         [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]]
_DP_B = [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84, 0]
_DP_E = [5179 / 57600, 0, 7571 / 16695, 393 / 640, -92097 / 339200, 187 / 2100, 1 / 40]


def _energy(p):
    return math.sqrt(1.0 + sum(v * v for v in p))


def _spinor(p, s, positron):
    """u_s(p) or v_s(p) = (1 +- p-slash) R_s / sqrt(2 p0 (p0 - p_x)), p-slash = beta p0 - beta alpha.p."""
    p0 = _energy(p)
    ps = _BETA * p0 - sum(_BETA @ _ALPHA[a] * p[a] for a in range(3))
    return (np.eye(4) + (-ps if positron else ps)) @ _R[s] / math.sqrt(2 * p0 * (p0 - p[0]))


def _apply(mat, v):
    """A constant 4 x 4 matrix on the component axis of [..., 4, nz, ny, nx]."""
    return torch.einsum("ab,...bzyx->...azyx", torch.as_tensor(mat, device="cuda"), v)


def _alpha_dot(k, v):
    """(alpha.k) v for three arrays (or numbers) k, componentwise on [..., 4, nz, ny, nx]."""
    a, b, c, d = (v[..., i, :, :, :] for i in range(4))
    km, kp = k[0] - 1j * k[1], k[0] + 1j * k[1]
    return torch.stack([k[2] * c + km * d, kp * c - k[2] * d, k[2] * a + km * b, kp * a - k[2] * b], dim=-4)


class _Grid:
    def __init__(self, n, L):
        self.n, self.L = n, L
        self.dx = [L[a] / n[a] if n[a] > 1 else 1.0 for a in range(3)]
        self.cell = self.dx[0] * self.dx[1] * self.dx[2]
        self.vol = math.prod(L[a] for a in range(3) if n[a] > 1)
        self.x, self.kap = [], []
        for a in range(3):
            shape = [n[a] if b == 2 - a else 1 for b in range(3)]
            x = -L[a] / 2 + torch.arange(n[a], device="cuda", dtype=_F64) * self.dx[a] if n[a] > 1 else torch.zeros(1, device="cuda", dtype=_F64)
            k = 2 * math.pi * torch.fft.fftfreq(n[a], self.dx[a], device="cuda", dtype=_F64) if n[a] > 1 else torch.zeros(1, device="cuda", dtype=_F64)
            self.x.append(x.reshape(shape))
            self.kap.append(k.reshape(shape))

    def on(self, mom):
        """Momenta along the non-trivial axes only."""
        return [mom[a] if self.n[a] > 1 else 0.0 for a in range(3)]

    def modes(self, K):
        return [self.kap[a] if self.n[a] > 1 else torch.full_like(self.kap[a], K[a]) for a in range(3)]

    def wave(self, mom):
        m = self.on(mom)
        return torch.exp(1j * (m[0] * self.x[0] + m[1] * self.x[1] + m[2] * self.x[2]))

    def transform(self, psi):
        """dx^d sum_x psi e^{-i kappa.x} on every mode."""
        ph = torch.exp(-1j * sum((self.kap[a] * self.x[a].flatten()[0] for a in range(3)), torch.zeros((), device="cuda", dtype=_F64)))
        return self.cell * ph * torch.fft.fftn(psi, dim=(-3, -2, -1))

    def at(self, psi, mom):
        return self.cell * (psi * self.wave([-v for v in mom])).sum(dim=(-3, -2, -1))


def _potential(d, g, t):
    """(component mu, A_mu(t, x))."""
    P, (X, Y, Z) = d["prm"], g.x
    if d["field"] == "sauter_gauss":
        return 1, P[0] / P[1] / math.cosh(P[1] * t)**2 * torch.exp(-(X * X + Y * Y + Z * Z) / P[2]**2)
    if d["field"] == "pulse_gauss":
        u = t - Y
        return 1, P[0] * torch.sin(P[1] * u) * torch.exp(-u * u / P[2]**2 - X * X / P[3]**2) + 0 * Z

    def one(x):
        return -(P[0] / P[2]) * torch.sin(P[2] * x) * torch.exp(-(P[1] * t)**2 - (P[2] * x)**2 - (P[3] * Y)**2 - (P[4] * Z)**2)
    return 0, one(X) if d["field"] == "single_e" else one(X + P[5]) + one(X - P[5])


class _Wave:
    """One marched wave: its background and its right-hand side (bg 0: U, 1: V)."""

    def __init__(self, d, g, bg):
        self.d, self.g, self.bg = d, g, bg
        self.mom = d["p"] if bg == 0 else d["q"]
        self.sp = torch.as_tensor(_spinor(self.mom, d["s"] if bg == 0 else d["r"], bg == 1), device="cuda").reshape(4, 1, 1, 1)
        self.K = [v if bg == 0 else -v for v in self.mom]
        self.plane = g.wave(self.K)
        self.k = g.modes(self.K)
        self.e = _energy(self.mom)

    def back(self, t):
        return self.sp * (np.exp((-1j if self.bg == 0 else 1j) * self.e * t) * self.plane)

    def source(self, t, y):
        mu, a = _potential(self.d, self.g, t)
        phi = a * (y + self.back(t))
        return -1j * (phi if mu == 0 else _apply(_ALPHA[mu - 1], phi))

    def rhs(self, t, y):
        s = torch.fft.fftn(y, dim=(-3, -2, -1))
        s = _alpha_dot(self.k, s) + _apply(_BETA, s)
        return -1j * torch.fft.ifftn(s, dim=(-3, -2, -1)) + self.source(t, y)


def _march(waves, hook=None):
    """Waves of one grid from 0 at t_out to t_in, fixed steps; hook(t, ys) is integrated along (its integral, or 0)."""
    d, g = waves[0].d, waves[0].g
    h, t0 = (d["t_in"] - d["t_out"]) / d["steps"], d["t_out"]
    y = [torch.zeros(4, g.n[2], g.n[1], g.n[0], device="cuda", dtype=torch.complex128) for _ in waves]
    k1, acc = [w.rhs(t0, v) for w, v in zip(waves, y)], 0.0
    g1 = hook(t0, y) if hook else 0.0
    for step in range(d["steps"]):
        t = t0 + step * h
        k, gs = [k1], [g1]
        for i in range(1, 7):
            ys = [v + h * sum(_DP_A[i][j] * k[j][w] for j in range(i) if _DP_A[i][j]) for w, v in enumerate(y)]
            k.append([w.rhs(t + _DP_C[i] * h, v) for w, v in zip(waves, ys)])
            gs.append(hook(t + _DP_C[i] * h, ys) if hook and (_DP_B[i] or i == 6) else 0.0)
        acc = acc + h * sum(b * v for b, v in zip(_DP_B, gs))
        y, k1, g1 = ys, k[6], gs[6]
    return y, acc


def _march_adaptive(waves, rtol=1e-5, atol=1e-10):
    """The waves of one call with one shared, controlled step."""
    d, g = waves[0].d, waves[0].g
    t, t_in, h = d["t_out"], d["t_in"], (d["t_in"] - d["t_out"]) / d["steps"]
    span = abs(t_in - t)
    y = [torch.zeros(4, g.n[2], g.n[1], g.n[0], device="cuda", dtype=torch.complex128) for _ in waves]
    k1 = [w.rhs(t, v) for w, v in zip(waves, y)]
    while abs(t_in - t) > 1e-12 * span:
        h = t_in - t if abs(h) > abs(t_in - t) else h
        k, err = [k1], 0.0
        for i in range(1, 7):
            ys = [v + h * sum(_DP_A[i][j] * k[j][w] for j in range(i) if _DP_A[i][j]) for w, v in enumerate(y)]
            k.append([w.rhs(t + _DP_C[i] * h, v) for w, v in zip(waves, ys)])
        for w in range(len(waves)):
            e = h * sum((b - c) * k[j][w] for j, (b, c) in enumerate(zip(_DP_B, _DP_E)) if b != c)
            sc = atol + rtol * torch.maximum(y[w].abs(), ys[w].abs())
            err = max(err, float(((e.abs() / sc)**2).mean().sqrt()))
        if err <= 1.0:
            t, y, k1 = t + h, ys, k[6]
        h *= 10.0 if err == 0 else min(10.0, max(0.2, 0.9 * err**-0.2))
    return y


def _marched(ds, g, bg, adaptive):
    if adaptive:
        return _march_adaptive([_Wave(d, g, bg) for d in ds])
    return [_march([_Wave(d, g, bg)])[0][0] for d in ds]


def _norm2(psi, g):
    return float(g.cell * (psi.abs()**2).sum())


def _spectrum64(psi, d, g):
    """C(m, (r, q)) for r = +1, -1 and every mode's positron q = -kappa: [2][nz][ny][nx]."""
    s = g.transform(psi)
    kap = g.modes(list(d["p"]))
    q = [-k for k in kap]
    q0 = torch.sqrt(1 + q[0]**2 + q[1]**2 + q[2]**2)
    out = []
    for r in (1, -1):
        R = torch.as_tensor(_R[r].astype(complex), device="cuda").reshape(4, 1, 1, 1)
        ps = _apply(_BETA, q0 * R - _alpha_dot(q, (R + 0 * q0)))
        out.append(torch.exp(1j * q0 * d["t_in"]) * (s.conj() * (R - ps)).sum(dim=0) / torch.sqrt(2 * q0 * (q0 - q[0])))
    return torch.stack(out)


def _project(v, k, sign):
    """P_sign(k) v = (v + sign H0 v / E) / 2 on [..., 4, nz, ny, nx]."""
    E = torch.sqrt(1 + k[0]**2 + k[1]**2 + k[2]**2)
    return 0.5 * (v + sign * (_alpha_dot(k, v) + _apply(_BETA, v)) / E)


def _project1(v, k, sign):
    H = sum(_ALPHA[a] * k[a] for a in range(3)) + _BETA
    return 0.5 * (v + sign * (H @ v) / _energy(k))


def _overlap_c(psi, d, g, q, r):
    return np.exp(1j * _energy(q) * d["t_in"]) * (g.at(psi, [-v for v in q]).conj().cpu().numpy() @ _spinor(q, r, True))


def _overlap_a(psi, d, g, p, s):
    return np.exp(1j * _energy(p) * d["t_in"]) * (_spinor(p, s, False).conj() @ g.at(psi, p).cpu().numpy())


def _solve64(ds, case):
    g = _Grid(ds[0]["n"], ds[0]["L"])
    U = _marched(ds, g, 0, case["adaptive"])
    V = _marched(ds, g, 1, case["adaptive"]) if case["full"] else [None] * len(ds)
    amp, prob, diag, spec = [], [], [], []
    for d, u, v in zip(ds, U, V):
        spec.append((_spectrum64(u, d, g).abs()**2).flatten())
        C = _overlap_c(u, d, g, d["q"], d["r"])
        if not case["full"]:
            C2 = _overlap_c(u, d, g, d["q"], -d["r"])
            amp.append([C, C2, 0, 0])
            prob.append([abs(C)**2, abs(C2)**2])
            diag.append([_norm2(u, g), 0.0])
            continue
        A = _overlap_a(v, d, g, d["p"], d["s"])
        su, sv, k = g.transform(u), g.transform(v), g.modes(list(d["p"]))
        B, D = (complex((su.conj() * _project(sv, k, sg)).sum()) / g.vol for sg in (1, -1))
        amp.append([C, D, A, B])
        prob.append([abs(C + D)**2, abs(A + B)**2])
        diag.append([_norm2(u, g), _norm2(v, g)])
    return {"amp": np.array(amp, complex), "prob": np.array(prob), "diag": np.array(diag), "spectrum": torch.cat(spec)}


def _pairs64(ds, case):
    ne, g = case["electrons"], _Grid(ds[0]["n"], ds[0]["L"])
    E, P, t = ds[:ne], ds[ne:], ds[0]["t_in"]
    U, V = torch.stack(_marched(E, g, 0, False)), torch.stack(_marched(P, g, 1, False))
    back_u = torch.stack([_Wave(d, g, 0).back(t) for d in E])
    back_v = torch.stack([_Wave(d, g, 1).back(t) for d in P])
    k = g.modes(list(E[0]["p"]))
    su, sv = g.transform(U), g.transform(V)

    def prod(a, b, s):
        return s * (a.reshape(len(a), -1).conj() @ b.reshape(len(b), -1).T)
    C, A = prod(U, back_v, g.cell), prod(back_u, V, g.cell)
    B, D = (prod(_project(su, k, sg), sv, 1 / g.vol) for sg in (1, -1))
    nu = (g.cell * (U.abs()**2).sum(dim=(1, 2, 3, 4)))[:, None].expand(len(E), len(P))
    nv = (g.cell * (V.abs()**2).sum(dim=(1, 2, 3, 4)))[None, :].expand(len(E), len(P))
    return {"amp": torch.stack([C, D, A, B], -1).reshape(-1, 4),
            "prob": torch.stack([(C + D).abs()**2, (A + B).abs()**2], -1).reshape(-1, 2),
            "diag": torch.stack([nu, nv], -1).reshape(-1, 2)}


def _ae(eps, v):
    return _alpha_dot([torch.tensor(float(e), device="cuda", dtype=_F64) for e in eps], v)


def _eps1(eps):
    return sum(_ALPHA[a] * eps[a] for a in range(3))


def _bw64(d, photons):
    """[n][4] amplitudes (ss, bs, sb, M) and the norms of U and V, for photons (k, eps) of one pair."""
    g = _Grid(d["n"], d["L"])
    wu, wv = _Wave(d, g, 0), _Wave(d, g, 1)
    partial = bool(d["flags"] & swf.BW_PARTIAL)
    p, q, t_in = d["p"], d["q"], d["t_in"]
    tabs = []
    for k, eps in photons:
        k0 = float(np.linalg.norm(k))
        shift = [int(round(k[a] * d["L"][a] / (2 * math.pi))) if g.n[a] > 1 else 0 for a in range(3)]
        roll = lambda v, sh=shift: torch.roll(v, (sh[2], sh[1], sh[0]), dims=(-3, -2, -1))  # noqa: E731
        one = torch.ones(g.n[2], g.n[1], g.n[0], device="cuda", dtype=_F64)
        ku = [v * one for v in wu.k]
        kv = [roll(v * one) for v in wv.k]
        x0 = [g.x[a].flatten()[0] if g.n[a] > 1 else 0.0 for a in range(3)]
        wrap = torch.exp(1j * sum((kv[a] + (k[a] if g.n[a] > 1 else 0.0) - (ku[a])) * x0[a] for a in range(2)))
        eu, ev = (torch.sqrt(1 + v[0]**2 + v[1]**2 + v[2]**2) for v in (ku, kv))
        tabs.append((k, eps, k0, roll, ku, kv, wrap, eu, ev, g.wave(k)))

    def ss_sum(tab, pairs):
        """sum over modes and signs of wrap (P x)^+ (alpha.eps) (P y) / Omega for pairs (x at U modes, y at V modes)."""
        k, eps, k0, roll, ku, kv, wrap, eu, ev, _ = tab
        tot = 0.0
        for x, y in pairs:
            for sg in (1, -1):
                px = _project(x, ku, sg).conj()
                for sp in (1, -1):
                    tot = tot + (wrap * (px * _ae(eps, _project(y, kv, sp))).sum(dim=0) / (sg * eu - sp * ev - k0)).sum()
        return complex(tot)

    def hook(t, ys):
        out = []
        if partial:
            du, dv = wu.source(t, ys[0]), wv.source(t, ys[1])
            su, sdu, sv, sdv = (g.transform(v) for v in (ys[0], du, ys[1], dv))
        ub, vb = wu.back(t), wv.back(t)
        for tab in tabs:
            k, eps, k0, roll = tab[:4]
            if not partial:
                ph = np.exp(-1j * k0 * t) * tab[9]
                out.append(torch.stack([g.cell * ((a.conj() * _ae(eps, b)).sum(dim=0) * ph).sum() for a, b in ((ys[0], ys[1]), (ub, ys[1]), (ys[0], vb))]))
                continue
            ss = 1j * np.exp(-1j * k0 * t) / g.vol * ss_sum(tab, ((sdu, roll(sv)), (su, roll(sdv))))
            kv1, ku1 = [p[a] - k[a] for a in range(3)], [k[a] - q[a] for a in range(3)]
            dvk, duk = g.at(dv, kv1).cpu().numpy(), g.at(du, ku1).cpu().numpy()
            ae, u, v = _eps1(eps), _spinor(p, d["s"], False), _spinor(q, d["r"], True)
            bs = sum(u.conj() @ ae @ _project1(dvk, kv1, sg) / (_energy(p) - sg * _energy(kv1) - k0) for sg in (1, -1))
            sb = sum(_project1(duk, ku1, sg).conj() @ ae @ v / (sg * _energy(ku1) + _energy(q) - k0) for sg in (1, -1))
            out.append(torch.tensor([ss, 1j * np.exp(1j * (_energy(p) - k0) * t) * bs, 1j * np.exp(1j * (_energy(q) - k0) * t) * sb], device="cuda"))
        return torch.stack(out)

    (U, V), acc = _march([wu, wv], hook)
    M = -acc.cpu().numpy()
    if not partial:
        su, sv = g.transform(U), g.transform(V)
        for j, tab in enumerate(tabs):
            k, eps, k0, roll = tab[:4]
            ek, ae = np.exp(-1j * k0 * t_in), _eps1(eps)
            M[j, 0] += ek / g.vol / 1j * ss_sum(tab, ((su, roll(sv)),))
            kv1, ku1 = [p[a] - k[a] for a in range(3)], [k[a] - q[a] for a in range(3)]
            vk, uk = g.at(V, kv1).cpu().numpy(), g.at(U, ku1).cpu().numpy()
            u, v = _spinor(p, d["s"], False), _spinor(q, d["r"], True)
            M[j, 1] += ek * np.exp(1j * _energy(p) * t_in) * sum(u.conj() @ ae @ _project1(vk, kv1, sg) / (1j * (_energy(p) - sg * _energy(kv1) - k0)) for sg in (1, -1))
            M[j, 2] += ek * np.exp(1j * _energy(q) * t_in) * sum(_project1(uk, ku1, sg).conj() @ ae @ v / (1j * (sg * _energy(ku1) + _energy(q) - k0)) for sg in (1, -1))
    return np.concatenate([M, M.sum(axis=1, keepdims=True)], axis=1), [_norm2(U, g), _norm2(V, g)]


def _layers(w):
    out, at = [], 0
    for i, o in ((6, 256), (256, 256), (256, 256), (256, 256), (256, 2)):
        out.append((w[at:at + i * o].reshape(o, i), w[at + i * o:at + i * o + o]))
        at += i * o + o
    return out


def _net64(w, x):
    norm = torch.as_tensor(_NORM, device="cuda", dtype=_F64)
    a = (x.to(_F64) - norm[:6]) * norm[6:12]
    for l, (W, b) in enumerate(_layers(w)):
        a = a @ W.T + b
        if l < 4:
            a = torch.nn.functional.gelu(a)
    return a, norm


def exact(case, seed):
    call = case["call"]
    if call == "forward":
        w = torch.as_tensor(_weights(seed), device="cuda", dtype=_F64)
        x, _ = _samples(case["rows"], seed)
        out = []
        for part in x.split(1 << 17):
            a, norm = _net64(w, part)
            out.append(torch.stack([a[:, 0] / norm[13] + norm[12], a[:, 1] - 2 * torch.log(norm[13])], dim=1))
        return torch.cat(out)
    if call == "train":
        w = torch.as_tensor(_weights(seed), device="cuda", dtype=_F64).requires_grad_()
        opt = torch.optim.Adam([w], lr=1e-3)
        x, y = _samples(case["batch"] * case["batches"], seed)
        for xb, yb in zip(x.split(case["batch"]), y.split(case["batch"])):
            a, norm = _net64(w, xb)
            r = (yb.to(_F64) - norm[12]) * norm[13] - a[:, 0]
            loss = 0.5 * (r * r * torch.exp(-a[:, 1]) + a[:, 1]).mean()
            opt.zero_grad()
            loss.backward()
            opt.step()
        return {"params": w.detach().cpu().numpy(), "loss": loss.detach().reshape(1)}
    ds = _dicts(case, seed)
    if case.get("adaptive") and case["prec"] == "c128":
        return None  # the step sequence decides the last digits
    if call in ("bw", "photons"):
        if call == "photons":
            k, eps, w = _photons(case, seed)
            if case["steps"] * len(k) * case["nx"] * case["ny"] > 1.5e8:
                return None
            amps, _ = _bw64(ds[0], list(zip(k, eps)))
            return {"amps": amps, "packet": (w[:, None] * amps).sum(axis=0)}
        if len(ds) * case["steps"] * (4 if case["partial"] else 1) > 600:
            return None
        got = [_bw64(d, [(d["k"], d["eps"])]) for d in ds]
        amp = np.concatenate([a for a, _ in got])
        return {"amp": amp, "prob": np.stack([np.abs(amp[:, 3])**2, np.zeros(len(ds))], axis=1), "diag": np.array([n for _, n in got])}
    if call == "pairs":
        return _pairs64(ds, case)
    if call == "solve":
        return _solve64(ds, case)
    g = _Grid(ds[0]["n"], ds[0]["L"])
    if call == "rhs":
        psi = torch.view_as_complex(_waves(case, seed)[0].to(_F64))
        return torch.view_as_real(_Wave(ds[0], g, 0).rhs(0.125, psi))
    if call == "spectrum":
        psi = torch.view_as_complex(_waves(case, seed).to(_F64))
        c = torch.stack([_spectrum64(v, d, g) for v, d in zip(psi, ds)])
        return {"c": torch.view_as_real(c).reshape(len(ds), 2, -1, 2), "prob": (c.abs()**2).reshape(len(ds), 2, -1)}
    return torch.view_as_real(torch.stack(_marched(ds, g, 0, case["adaptive"])))
