"""Measured work of the WENO5-CT MHD library: what a program that uses it has
it do, through the public entry points, over the range it is used in.

A case is one of four kinds of program:

``step``    one periodic box: load a state, take steps, read the state back;
``batch``   many independent uneven boxes in one context, replayed steps;
``adjoint`` the gradient of a rollout misfit (torch.autograd);
``monitor`` the diagnostics a run prints between steps.

Inputs are made on the GPU from the seed alone: solenoidal k^-5/3 velocities
and divergence-free field perturbations (the benchmark's turbulence), small
linear waves, a blast, or an Alfven wave with an overpressure.  A box of the
FP32-bulk form is handed back in float (what a run of that precision keeps of
a snapshot), one of the FP64 forms in double.

`exact` is the scheme of the paper (WENO5 / WENO5-Z characteristic fluxes,
transport-flux constrained transport, RK4, CFL step) in plain torch double
precision, written out field by field, with torch.autograd for the gradients.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1812_04278_gb300 import adjoint, w5ct

GAMMA = 5.0 / 3.0
# flops of one zone's RK4 + CT step and of one step's vector-Jacobian product
FLOPS = {"z": 36057, "js": 34881}
FLOPS_VJP = 132768
PRECISION = {"fp64": w5ct.W5CT_FP64, "fp32": w5ct.W5CT_FP32_BULK, "dw": w5ct.W5CT_FP64_DW}
PATCH_SIZES = (16, 24, 32, 48, 64)


def listed():
    return [
        # linear-wave convergence and regression runs: tiny boxes, many steps, where launches and latency count
        _step("wave32_fp64", "wave", 32, 32, 32, "fp64", "z", steps=2),
        # the same in the fast form: the shortest calls a user makes
        _step("turb32_fp32", "turb", 32, 32, 32, "fp32", "z", steps=2),
        # a production box that no tile divides, WENO5 with floors, host output and totals after the step
        _step("ragged_fp64_js", "turb", 100, 70, 50, "fp64", "js", floors=True, host=True),
        # medium turbulence box with double-word weights
        _step("turb128_dw", "turb", 128, 128, 128, "dw", "z"),
        # the headline turbulence box in both arithmetic forms
        _step("turb256_fp64", "turb", 256, 256, 256, "fp64", "z"),
        _step("turb256_fp32", "turb", 256, 256, 256, "fp32", "z", steps=2),
        # the largest run: blast in supersonic turbulence, WENO5 with floors
        _step("blast512_fp32_js", "blast", 512, 512, 512, "fp32", "js", floors=True),
        # an ensemble of uneven boxes advanced together by graph replay
        _batch("batch512_fp32", 512, 1803, "fp32", "z", steps=3),
        # a smaller ensemble in double with one dt for all
        _batch("batch48_fp64", 48, 1804, "fp64", "z", steps=1, graph=False),
        # gradients for inversion / data assimilation
        _adjoint("adjoint64_fp64", 64, 64, 64, "fp64", "z", 2),
        _adjoint("adjoint64_fp32", 64, 64, 64, "fp32", "js", 3),
        # what a run prints between steps
        {"name": "monitor256_fp64", "kind": "monitor", "nx": 256, "ny": 256, "nz": 256, "precision": "fp64"},
    ]


def _step(name, state, nx, ny, nz, precision, weno, steps=1, floors=False, host=False):
    return {"name": name, "kind": "step", "state": state, "nx": nx, "ny": ny, "nz": nz, "precision": precision,
            "weno": weno, "steps": steps, "floors": floors, "host": host}


def _batch(name, npatch, sizes_seed, precision, weno, steps, graph=True, odd=False):
    return {"name": name, "kind": "batch", "npatch": npatch, "sizes_seed": sizes_seed, "odd": odd,
            "precision": precision, "weno": weno, "steps": steps, "graph": graph}


def _adjoint(name, nx, ny, nz, precision, weno, steps):
    return {"name": name, "kind": "adjoint", "nx": nx, "ny": ny, "nz": nz, "precision": precision, "weno": weno,
            "steps": steps}


def draw(rng):
    """One more case: sizes spread over their logarithm from 8 cells an axis
    to the listed largest, every precision and weight variant."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("step", "step", "step", "step", "batch", "adjoint", "monitor"))
    if kind == "step":
        precision = rng.choice(("fp64", "fp32", "fp32", "dw"))
        top, most = (512, 1 << 26) if precision == "fp32" else (256, 1 << 23)
        while True:
            n = [size(8, top) for _ in range(3)]
            if n[0] * n[1] * n[2] <= most:
                break
        floors = rng.random() < 0.3
        c = _step("", rng.choice(("turb", "turb", "wave")), *n, precision, rng.choice(("z", "z", "js")), rng.choice((1, 2)),
                  floors, n[0] * n[1] * n[2] <= 1 << 19 and rng.random() < 0.3)
    elif kind == "batch":
        precision = rng.choice(("fp32", "fp32", "fp64"))
        c = _batch("", size(4, 400 if precision == "fp32" else 40), rng.randrange(1 << 20), precision,
                   rng.choice(("z", "js")), rng.choice((1, 2)), rng.random() < 0.5, rng.random() < 0.5)
    elif kind == "adjoint":
        precision = rng.choice(("fp64", "fp32"))
        c = _adjoint("", *(size(10, 64) for _ in range(3)), precision, "z" if precision == "fp64" else "js",
                     rng.choice((1, 2, 3)))
    else:
        c = {"kind": "monitor", "nx": size(16, 256), "ny": size(16, 256), "nz": size(16, 256),
             "precision": rng.choice(("fp64", "fp32"))}
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs

DIM = (-1, -2, -3)      # tensor dimension of the x, y and z axes: arrays are (..., nz, ny, nx)


def _gen(seed, *more):
    g = torch.Generator(device="cuda")
    g.manual_seed(hash((int(seed),) + more) & 0x7FFFFFFF)
    return g


def _at(a, axis, s):
    """a at index + s along an axis, periodic."""
    return torch.roll(a, -s, DIM[axis])


def _modes(shape, kmax, slope, g):
    """Solenoidal Gaussian random-phase coefficients with |F| ~ |k|^slope for
    1.5 < |k| <= kmax on the cube of low wave numbers, and that cube's k."""
    k = torch.arange(-kmax, kmax + 1, dtype=torch.float64, device="cuda")
    KZ, KY, KX = torch.meshgrid(k, k, torch.arange(0, kmax + 1, dtype=torch.float64, device="cuda"), indexing="ij")
    K2 = KX * KX + KY * KY + KZ * KZ
    amp = torch.where((K2 > 2.25) & (K2 <= kmax * kmax), K2.clamp(min=1.0) ** (0.5 * slope), torch.zeros_like(K2))
    F = torch.randn((3,) + K2.shape + (2,), generator=g, dtype=torch.float64, device="cuda")
    F = torch.view_as_complex(F) * amp
    kd = (KX * F[0] + KY * F[1] + KZ * F[2]) / K2.clamp(min=1.0)
    return torch.stack([F[0] - KX * kd, F[1] - KY * kd, F[2] - KZ * kd]), (KX, KY, KZ)


def _field(F, K, shape, shift):
    """The real field of the coefficients F, sampled `shift` cells from the centres."""
    nx, ny, nz = shape
    ph = 2.0 * math.pi * (K[0] * (shift[0] / nx) + K[1] * (shift[1] / ny) + K[2] * (shift[2] / nz))
    C = F * torch.polar(torch.ones_like(ph), ph)
    m = F.shape[-1] - 1
    S = torch.zeros((nz, ny, nx // 2 + 1), dtype=torch.complex128, device="cuda")
    iz = torch.arange(-m, m + 1, device="cuda") % nz
    iy = torch.arange(-m, m + 1, device="cuda") % ny
    S[iz[:, None, None], iy[None, :, None], torch.arange(m + 1, device="cuda")[None, None, :]] = C
    return torch.fft.irfftn(S, s=(nz, ny, nx))


def _curl(A, dx):
    """Face fields b = curl A of an edge vector potential."""
    bx = (A[2] - _at(A[2], 1, -1)) / dx[1] - (A[1] - _at(A[1], 2, -1)) / dx[2]
    by = (A[0] - _at(A[0], 2, -1)) / dx[2] - (A[2] - _at(A[2], 0, -1)) / dx[0]
    bz = (A[1] - _at(A[1], 0, -1)) / dx[0] - (A[0] - _at(A[0], 1, -1)) / dx[1]
    return torch.stack([bx, by, bz])


def _centre6(b):
    """Sixth-order face-to-centre interpolation of the initial state."""
    w = (3.0, -25.0, 150.0, 150.0, -25.0, 3.0)
    return torch.stack([sum(w[o + 3] / 256.0 * _at(b[a], a, o) for o in range(-3, 3)) for a in range(3)])


def _conserved(rho, v, P, b):
    Bc = _centre6(b)
    E = P / (GAMMA - 1.0) + 0.5 * rho * (v * v).sum(0) + 0.5 * (Bc * Bc).sum(0)
    return torch.stack([rho, rho * v[0], rho * v[1], rho * v[2], E])


EDGE = ((0.0, 0.5, 0.5), (0.5, 0.0, 0.5), (0.5, 0.5, 0.0))


def _turbulence(shape, g, mach, beta, P0, B_dir, kmax, texture=0.0):
    """(cons, bface): uniform rho and P (or textured), solenoidal k^-5/3
    velocity at rms Mach `mach`, mean field of plasma beta `beta` along B_dir
    and a 10% divergence-free perturbation."""
    nx, ny, nz = shape
    B0 = math.sqrt(2.0 * P0 / beta)
    F, K = _modes(shape, kmax, -11.0 / 6.0, g)
    v = torch.stack([_field(F[c], K, shape, (0.0, 0.0, 0.0)) for c in range(3)])
    v *= mach * math.sqrt(GAMMA * P0) / (v * v).sum(0).mean().sqrt()
    F, K = _modes(shape, kmax, -17.0 / 6.0, g)
    b = _curl([_field(F[c], K, shape, EDGE[c]) for c in range(3)], (1.0 / nx, 1.0 / ny, 1.0 / nz))
    b *= 0.1 * B0 / (b * b).sum(0).mean().sqrt()
    norm = math.sqrt(sum(d * d for d in B_dir))
    for a in range(3):
        b[a] += B0 * B_dir[a] / norm
    rho = torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda")
    return _conserved(rho, v, torch.full_like(rho, P0), b), b


def _kmax(shape):
    return max(2, min(32, min(shape) // 8))


def _state(case, seed):
    """Initial (cons, bface) of a box."""
    shape = (case["nx"], case["ny"], case["nz"])
    g = _gen(seed, 1)
    kind = case.get("state", "turb")
    if kind == "wave":
        # linear waves of amplitude 1e-6 on rho = P = 1, B = (1, sqrt 2, 1/2)
        cons, b = _turbulence(shape, g, 1e-6, 2.0, 1.0, (1.0, 2.0 ** 0.5, 0.5), min(3, _kmax(shape) + 1))
        mean = b.mean((1, 2, 3), keepdim=True)
        b = mean + 1e-5 * (b - mean)
        rho = torch.ones_like(cons[0])
        return _conserved(rho, cons[1:4], rho, b), b
    if kind == "blast":
        # P = 100 inside r = 0.05 of an ambient 0.1, beta 0.2, Mach-5 turbulence
        cons, b = _turbulence(shape, g, 5.0, 0.2, 0.1, (1.0, 1.0, 1.0), _kmax(shape))
        x, y, z = ((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n - 0.5 for n in shape)
        r2 = (x * x)[None, None, :] + (y * y)[None, :, None] + (z * z)[:, None, None]
        cons[4] += torch.where(r2 < 0.05 ** 2, 99.9 / (GAMMA - 1.0), 0.0)
        return cons, b
    return _turbulence(shape, g, 1.0, 1.0, 1.0 / GAMMA, (1.0, 0.0, 0.0), _kmax(shape))


def _patches(case):
    """The sizes of a batch: each axis drawn from the ensemble's sizes, or any
    size of their range."""
    r = np.random.RandomState(case["sizes_seed"])
    if case["odd"]:
        return [tuple(int(round(v)) for v in np.exp(r.uniform(np.log(10), np.log(64), 3))) for _ in range(case["npatch"])]
    return [tuple(int(v) for v in r.choice(PATCH_SIZES, 3)) for _ in range(case["npatch"])]


def _patch_state(shape, seed, p):
    """One patch's turbulence: its own rms Mach 0.5-3, beta 0.1-10, mean field direction."""
    r = np.random.RandomState((int(seed) * 7919 + p) & 0x7FFFFFFF)
    return _turbulence(shape, _gen(seed, 2, p), r.uniform(0.5, 3.0), math.exp(r.uniform(math.log(0.1), math.log(10.0))),
                       1.0 / GAMMA, tuple(r.standard_normal(3)), _kmax(shape))


def _alfven(case, seed):
    """(rho, v, P, A, B0) of an oblique circularly polarised Alfven wave of
    amplitude 0.1 with a Gaussian overpressure, rho and P textured by 2%."""
    shape = nx, ny, nz = case["nx"], case["ny"], case["nz"]
    ph = torch.rand(9, generator=_gen(seed, 3), dtype=torch.float64, device="cuda") * 2.0 * math.pi
    tp = 2.0 * math.pi
    kvec = (tp, 2.0 * tp, 2.0 * tp)
    e1, e2 = (-2.0 / 5 ** 0.5, 1.0 / 5 ** 0.5, 0.0), (-2.0 / 45 ** 0.5, -4.0 / 45 ** 0.5, 5.0 / 45 ** 0.5)

    def xyz(s):
        x, y, z = ((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5 + o) / n for n, o in zip(shape, s))
        return x[None, None, :], y[None, :, None], z[:, None, None]

    def phase(s):
        x, y, z = xyz(s)
        return kvec[0] * x + kvec[1] * y + kvec[2] * z + ph[0]

    p = phase((0.0, 0.0, 0.0))
    x, y, z = xyz((0.0, 0.0, 0.0))
    v = torch.stack([0.1 * (e1[c] * torch.sin(p) + e2[c] * torch.cos(p)) for c in range(3)])
    A = torch.stack([0.1 / (3.0 * tp) * (e1[c] * torch.sin(phase(EDGE[c])) + e2[c] * torch.cos(phase(EDGE[c])))
                     for c in range(3)])
    r2 = (x - 0.5) ** 2 + (y - 0.5) ** 2 + (z - 0.5) ** 2
    rho = 1.0 + 0.02 * (torch.sin(tp * x + ph[1]) * torch.cos(tp * y + ph[2]) + 0.5 * torch.sin(tp * z + ph[3]))
    P = 0.1 * (1.0 + 9.0 * torch.exp(-r2 / 0.01)) * (1.0 + 0.02 * torch.cos(tp * y + ph[4]) * torch.sin(tp * z + ph[5])
                                                     + 0.01 * torch.sin(tp * x + ph[6]))
    return rho, v, P, A, (1.0 / 3.0, 2.0 / 3.0, 2.0 / 3.0)


def _adjoint_dt(case):
    return 0.12 / max(case["nx"], case["ny"], case["nz"])


# ---------------------------------------------------------------- the program


def _config(case):
    return w5ct.make_config(precision=PRECISION[case["precision"]],
                            weno_variant=w5ct.W5CT_WENO_JS if case.get("weno") == "js" else w5ct.W5CT_WENO_Z,
                            floors=int(case.get("floors", False) or case["kind"] == "batch"))


def prepare(case, seed):
    stream = torch.cuda.current_stream().cuda_stream
    s = {"case": case}
    if case["kind"] == "batch":
        shapes = _patches(case)
        n = [a * b * c for a, b, c in shapes]
        cells = sum(n)
        s["cons"] = torch.empty(5 * cells, dtype=torch.float64, device="cuda")
        s["bface"] = torch.empty(3 * cells, dtype=torch.float64, device="cuda")
        s["parts"], at = [], 0
        for p, sh in enumerate(shapes):
            c, b = _patch_state(sh, seed, p)
            s["cons"][5 * at:5 * (at + n[p])] = c.reshape(-1)
            s["bface"][3 * at:3 * (at + n[p])] = b.reshape(-1)
            s["parts"].append((slice(5 * at, 5 * (at + n[p])), slice(3 * at, 3 * (at + n[p]))))
            at += n[p]
        s["out"] = torch.empty_like(s["cons"]), torch.empty_like(s["bface"])
        s["batch"] = w5ct.Batch(shapes, [tuple(1.0 / v for v in sh) for sh in shapes], _config(case), stream=stream)
        return s
    shape = (case["nx"], case["ny"], case["nz"])
    dx = tuple(1.0 / v for v in shape)
    if case["kind"] == "adjoint":
        rho, v, P, A, B0 = _alfven(case, seed)
        s["leaves"] = [t.clone().requires_grad_(True) for t in (rho, v, A)]
        s["P"], s["B0"] = P, B0
        s["target"] = _target(case, seed)
    else:
        s["cons"], s["bface"] = _state(case, seed)
        s["out"] = torch.empty_like(s["cons"]), torch.empty_like(s["bface"])
    torch.cuda.empty_cache()
    s["solver"] = w5ct.Solver(shape, dx, _config(case), stream=stream)
    if case["kind"] == "monitor":
        s["solver"].set_state(s["cons"], s["bface"])
        s["dx"] = dx
    return s


def _target(case, seed):
    """The observed state of the misfit: a shifted wave of the same kind."""
    rho, v, P, A, B0 = _alfven(case, int(seed) + 7001)
    b = _curl(A, tuple(1.0 / case[n] for n in ("nx", "ny", "nz")))
    b = torch.stack([b[a] + B0[a] for a in range(3)])
    return _conserved(rho, v, P, b), b


def run(s):
    case = s["case"]
    single = case["precision"] == "fp32"
    if case["kind"] == "batch":
        b = s["batch"]
        for p, (c, f) in enumerate(s["parts"]):
            b.set_state(p, s["cons"][c], s["bface"][f])
        if case["graph"]:
            b.step_graph(case["steps"])
        else:
            for _ in range(case["steps"]):
                b.step_cfl()
        for p, (c, f) in enumerate(s["parts"]):
            w5ct.w5ct_get_state(b.ctx, s["out"][0][c], s["out"][1][f], None, 1, patch=p)
        return [t.float() if single else t for t in s["out"]]
    if case["kind"] == "adjoint":
        rho, v, A = s["leaves"]
        L = adjoint.rollout_misfit(rho, v, A, s["solver"], s["P"], s["B0"], *s["target"], _adjoint_dt(case), case["steps"])
        out = [L.detach(), *torch.autograd.grad(L, (rho, v, A))]
        return [t.float() if single else t for t in out]
    sol = s["solver"]
    if case["kind"] == "monitor":
        return [sol.max_signal_speed(), sol.cfl_dt(), np.array(sol.div_b_norm()), sol.conserved_totals(),
                w5ct.w5ct_conserved_totals_noalloc(s["cons"], s["bface"], sol.shape, sol.dx,
                                                   torch.cuda.current_stream().cuda_stream)]
    sol.set_state(s["cons"], s["bface"])
    for _ in range(case["steps"]):
        sol.step_cfl()
    if case["host"]:
        cons, bface, _ = sol.get_state()
        out = [cons, bface, sol.conserved_totals()]
        return [t.astype(np.float32) if single else t for t in out]
    w5ct.w5ct_get_state(sol.ctx, *s["out"], None, 1)
    return [t.float() if single else t for t in s["out"]]


def work(case):
    if case["kind"] == "batch":
        cells = sum(a * b * c for a, b, c in _patches(case))
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
    out = 4 if case["precision"] == "fp32" else 8
    if case["kind"] == "monitor":
        return {"bytes": cells * 8 * 8, "flops": cells * 200}
    if case["kind"] == "adjoint":
        # rho, v, P, A and the target in, seven gradient planes out
        return {"bytes": cells * (16 * 8 + 7 * out), "flops": cells * case["steps"] * (FLOPS[case["weno"]] + FLOPS_VJP)}
    return {"bytes": cells * 8 * (8 + out), "flops": cells * case["steps"] * FLOPS[case["weno"]]}


# ---------------------------------------------------------------- 64-bit values


def _centre4(b):
    return [(9.0 * (_at(b[a], a, -1) + b[a]) - (_at(b[a], a, -2) + _at(b[a], a, 1))) / 16.0 for a in range(3)]


def _primitives(q, B, floors):
    rho = q[0].clamp(min=1e-8) if floors else q[0]
    v = [q[1] / rho, q[2] / rho, q[3] / rho]
    P = (GAMMA - 1.0) * (q[4] - 0.5 * rho * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2) - 0.5 * (B[0] ** 2 + B[1] ** 2 + B[2] ** 2))
    return rho, v, P.clamp(min=1e-8) if floors else P


def _speeds(rho, P, Bn, B1, B2):
    """c_s^2, c_f^2, c_slow^2, c_f^2 - c_s^2, c_s^2 - c_slow^2 without cancellation."""
    cs2, ca2, bt2 = GAMMA * P / rho, Bn * Bn / rho, (B1 * B1 + B2 * B2) / rho
    sd = torch.sqrt((cs2 - ca2) ** 2 + bt2 * (bt2 + 2.0 * ca2 + 2.0 * cs2))
    a = ca2 + bt2 - cs2
    big = 0.5 * (sd + a.abs())
    oth = cs2 * bt2 / big
    fmc, cms = torch.where(a >= 0, big, oth), torch.where(a >= 0, oth, big)
    cf2 = cs2 + fmc
    return cs2, cf2, cs2 * ca2 / cf2, fmc, cms


def _phi(a, b, c, d, js):
    i0 = 13.0 * (a - b) ** 2 + 3.0 * (a - 3.0 * b) ** 2
    i1 = 13.0 * (b - c) ** 2 + 3.0 * (b + c) ** 2
    i2 = 13.0 * (c - d) ** 2 + 3.0 * (3.0 * c - d) ** 2
    if js:
        a0, a1, a2 = 1.0 / (1e-6 + i0) ** 2, 6.0 / (1e-6 + i1) ** 2, 3.0 / (1e-6 + i2) ** 2
    else:
        t = (i0 - i2).abs()
        a0, a1, a2 = 1.0 + (t / (1e-40 + i0)) ** 2, 6.0 + 6.0 * (t / (1e-40 + i1)) ** 2, 3.0 + 3.0 * (t / (1e-40 + i2)) ** 2
    D = a0 + a1 + a2
    return a0 / D / 3.0 * (a - 2.0 * b + c) + (a2 / D - 0.5) / 6.0 * (b - 2.0 * c + d)


def _sweep(ax, js, floors, *fields):
    """Face fluxes along one axis at the forward faces of every cell: rho, the
    lab momenta, E, and the two transport fluxes of the tangential fields."""
    q, B = fields[:5], fields[5:]
    n, t1, t2 = ax, (ax + 1) % 3, (ax + 2) % 3
    r, v, P = _primitives(q, B, floors)
    vn, v1, v2, Bn, B1, B2 = v[n], v[t1], v[t2], B[n], B[t1], B[t2]
    Ps = P + 0.5 * (Bn * Bn + B1 * B1 + B2 * B2)
    F = [r * vn, r * vn * vn + Ps - Bn * Bn, r * vn * v1 - Bn * B1, r * vn * v2 - Bn * B2, B1 * vn - Bn * v1,
         B2 * vn - Bn * v2, (q[4] + Ps) * vn - Bn * (vn * Bn + v1 * B1 + v2 * B2)]
    U = [q[0], q[1 + n], q[1 + t1], q[1 + t2], B1, B2, q[4]]
    _, cf2, cl2, _, _ = _speeds(r, P, Bn, B1, B2)
    speed = [torch.sqrt(cf2), Bn.abs() / torch.sqrt(r), torch.sqrt(cl2)]
    lam = [vn - speed[0], vn - speed[1], vn - speed[2], vn, vn + speed[2], vn + speed[1], vn + speed[0]]
    alpha = [torch.maximum(l.abs(), _at(l, ax, 1).abs()) for l in lam]
    bv1, bv2 = (0.5 * (Bn * w + _at(Bn * w, ax, 1)) for w in (v1, v2))

    # Appendix A at the mean of the two cells' primitives
    r, vn, v1, v2, Bn, B1, B2, P = (0.5 * (w + _at(w, ax, 1)) for w in (r, vn, v1, v2, Bn, B1, B2, P))
    cs2, cf2, cl2, fmc, cms = _speeds(r, P, Bn, B1, B2)
    cs, cf, cl = torch.sqrt(cs2), torch.sqrt(cf2), torch.sqrt(cl2)
    one = torch.ones_like(r)
    dfs = fmc + cms
    apart = torch.sqrt(dfs) >= 1e-30
    af, as_ = (torch.where(apart, torch.sqrt((w / torch.where(apart, dfs, one)).clamp(min=0.0)), one) for w in (cms, fmc))
    bt = B1 * B1 + B2 * B2
    some = bt > 1e-30
    m = torch.sqrt(torch.where(some, bt, one))
    b1, b2 = (torch.where(some, w / m, one * 0.5 ** 0.5) for w in (B1, B2))
    sg = torch.where(Bn >= 1e-30, one, -one)
    g1, g2, vv, sr, bv = GAMMA - 1.0, (GAMMA - 2.0) / (GAMMA - 1.0), vn * vn + v1 * v1 + v2 * v2, torch.sqrt(r), b1 * v1 + b2 * v2
    Gf, Ga, Gs = af * cf * vn - as_ * cl * sg * bv, sg * (b2 * v1 - b1 * v2), as_ * cl * vn + af * cf * sg * bv
    pre, tau = 0.5 / cs2, g1 / cs2
    flux = [0.0] * 7
    for m_, s in enumerate((1, 1, 1, 0, -1, -1, -1)):
        if m_ in (0, 6):
            L = [pre * (0.5 * g1 * af * vv + s * Gf), pre * (-g1 * af * vn - s * af * cf), pre * (-g1 * af * v1 + s * cl * as_ * b1 * sg),
                 pre * (-g1 * af * v2 + s * cl * as_ * b2 * sg), pre * (-g1 * af * B1 + sr * cs * as_ * b1),
                 pre * (-g1 * af * B2 + sr * cs * as_ * b2), pre * g1 * af]
            R = [af, af * (vn - s * cf), af * v1 + s * cl * as_ * b1 * sg, af * v2 + s * cl * as_ * b2 * sg, cs * as_ * b1 / sr,
                 cs * as_ * b2 / sr, af * (0.5 * vv + cf2 - g2 * cs2) - s * Gf]
        elif m_ in (1, 5):
            L = [0.5 * Ga, None, -0.5 * b2 * sg, 0.5 * b1 * sg, -s * 0.5 * sr * b2, s * 0.5 * sr * b1, None]
            R = [None, None, -b2 * sg, b1 * sg, -s * b2 / sr, s * b1 / sr, -Ga]
        elif m_ in (2, 4):
            L = [pre * (0.5 * g1 * as_ * vv + s * Gs), pre * (-g1 * as_ * vn - s * as_ * cl), pre * (-g1 * as_ * v1 - s * cf * af * b1 * sg),
                 pre * (-g1 * as_ * v2 - s * cf * af * b2 * sg), pre * (-g1 * as_ * B1 - sr * cs * af * b1),
                 pre * (-g1 * as_ * B2 - sr * cs * af * b2), pre * g1 * as_]
            R = [as_, as_ * (vn - s * cl), as_ * v1 - s * cf * af * b1 * sg, as_ * v2 - s * cf * af * b2 * sg, -cs * af * b1 / sr,
                 -cs * af * b2 / sr, as_ * (0.5 * vv + cl2 - g2 * cs2) - s * Gs]
        else:
            L = [1.0 - 0.5 * tau * vv, tau * vn, tau * v1, tau * v2, tau * B1, tau * B2, -tau]
            R = [one, vn, v1, v2, None, None, 0.5 * vv]
        proj = [[sum(l * _at(x, ax, k) for l, x in zip(L, X) if l is not None) for k in range(-2, 4)] for X in (F, U)]
        f, u = proj
        plus = [0.5 * ((f[j + 1] - f[j]) + alpha[m_] * (u[j + 1] - u[j])) for j in range(5)]
        minus = [0.5 * ((f[j + 1] - f[j]) - alpha[m_] * (u[j + 1] - u[j])) for j in range(5)]
        w = (7.0 * (f[2] + f[3]) - f[1] - f[4]) / 12.0 - _phi(*plus[:4], js) + _phi(*minus[:0:-1], js)
        flux = [x if y is None else x + w * y for x, y in zip(flux, R)]
    mom = [None] * 3
    mom[n], mom[t1], mom[t2] = flux[1], flux[2], flux[3]
    return (flux[0], *mom, flux[6], flux[4] + bv1, flux[5] + bv2)


def _rhs(q, b, dx, js, floors, grad):
    B = _centre4(b)
    D, S = [0.0] * 5, []
    for ax in range(3):
        if grad:
            f = checkpoint(_sweep, ax, js, floors, *q, *B, use_reentrant=False)
        else:
            f = _sweep(ax, js, floors, *q, *B)
        D = [d - (f[i] - _at(f[i], ax, -1)) / dx[ax] for i, d in enumerate(D)]
        S.append(f[5:])
    (fy, fz), (gz, gx), (hx, hy) = S
    O = [0.5 * (gx + _at(gx, 0, 1)) - 0.5 * (fy + _at(fy, 1, 1)), 0.5 * (hy + _at(hy, 1, 1)) - 0.5 * (gz + _at(gz, 2, 1)),
         0.5 * (fz + _at(fz, 2, 1)) - 0.5 * (hx + _at(hx, 0, 1))]
    return D, O


def _ct(b, O, f, dx):
    def d(o, a):
        return (o - _at(o, a, -1)) / dx[a]
    return [b[0] + f * (d(O[2], 2) - d(O[0], 1)), b[1] + f * (d(O[0], 0) - d(O[1], 2)), b[2] + f * (d(O[1], 1) - d(O[2], 0))]


def _rk4(q, b, dt, dx, js, floors, grad=False):
    qs, bs, Dsum, Osum = q, b, [0.0] * 5, [0.0] * 3
    for c, w in ((0.5, 1.0 / 6.0), (0.5, 1.0 / 3.0), (1.0, 1.0 / 3.0), (0.0, 1.0 / 6.0)):
        D, O = _rhs(qs, bs, dx, js, floors, grad)
        Dsum, Osum = [x + w * y for x, y in zip(Dsum, D)], [x + w * y for x, y in zip(Osum, O)]
        if c:
            qs, bs = [x + c * dt * y for x, y in zip(q, D)], _ct(b, O, c * dt, dx)
    return [x + dt * y for x, y in zip(q, Dsum)], _ct(b, Osum, dt, dx)


def _signal(q, b, floors):
    B = _centre4(b)
    r, v, P = _primitives(q, B, floors)
    return [float((v[a].abs() + torch.sqrt(_speeds(r, P, B[a], B[(a + 1) % 3], B[(a + 2) % 3])[1])).max()) for a in range(3)]


def _advance(cons, b, dx, case):
    js, floors = case["weno"] == "js", bool(case.get("floors", False) or case["kind"] == "batch")
    q, b = list(cons), list(b)
    for _ in range(case["steps"]):
        q, b = _rk4(q, b, 0.8 / sum(S / h for S, h in zip(_signal(q, b, floors), dx)), dx, js, floors)
    return torch.stack(q), torch.stack(b)


def exact(case, seed):
    if case["kind"] == "batch":
        shapes = _patches(case)
        if len(shapes) * case["steps"] > 60:
            return None     # minutes of small launches
        got = [_advance(*_patch_state(sh, seed, p), tuple(1.0 / v for v in sh), case) for p, sh in enumerate(shapes)]
        return [torch.cat([g[i].reshape(-1) for g in got]) for i in range(2)]
    dx = tuple(1.0 / case[n] for n in ("nx", "ny", "nz"))
    cells = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "adjoint":
        rho, v, P, A, B0 = _alfven(case, seed)
        rho, v, A = (t.clone().requires_grad_(True) for t in (rho, v, A))
        b = _curl(A, dx)
        b = torch.stack([b[a] + B0[a] for a in range(3)])
        q, b = list(_conserved(rho, v, P, b)), list(b)
        for _ in range(case["steps"]):
            q, b = _rk4(q, b, _adjoint_dt(case), dx, case["weno"] == "js", False, grad=True)
        tq, tb = _target(case, seed)
        L = 0.5 * dx[0] * dx[1] * dx[2] * (((torch.stack(q) - tq) ** 2).sum() + ((torch.stack(b) - tb) ** 2).sum())
        return [L.detach(), *torch.autograd.grad(L, (rho, v, A))]
    cons, b = _state(case, seed)
    if case["kind"] == "monitor":
        S = _signal(list(cons), list(b), False)
        total = torch.cat([cons, b]).sum((1, 2, 3)).cpu().numpy() * dx[0] * dx[1] * dx[2]
        # the divergence of a divergence-free field is rounding: it has no value
        return [np.array(S), 0.8 / sum(s / h for s, h in zip(S, dx)), None, total, total]
    if cells > 1 << 25:
        return None         # its intermediate planes alone would fill the card
    q, b = _advance(cons, b, dx, case)
    if not case["host"]:
        return [q, b]
    total = torch.cat([q, b]).sum((1, 2, 3)).cpu().numpy() * dx[0] * dx[1] * dx[2]
    return [q.cpu().numpy(), b.cpu().numpy(), total]
