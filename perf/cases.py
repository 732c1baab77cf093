"""What a user of the library has it do, as cases that can be timed and compared.

The paths are the ones the README's example walks through and the configurations of the benchmark
name: the split step in float32 and float64 from one small field to 1024^3, the ragged ensemble,
the adjoint of a run, the diagnostics, the analysis of a snapshot (structure functions and
helicity), the imaginary-time preparation and the vortex-ring start field.

    listed()            the cases that are always measured
    draw(rng)           one more case of the same ranges
    prepare(case, seed) the plan, the fields and the parameters a program holds before the call
    run(state)          one pass through the public entry points, and its outputs
    work(case)          bytes and flops the pass cannot do without
    exact(case, seed)   the same outputs in 64 bits by plain torch on the same inputs

Inputs are made by torch from the seed alone (no field generator of the library is used except
where the generator is the case).  Fields: smoothed random phases (Gaussian low modes, RMS pi) and
products of tanh-core vortex rings, the two start fields of the configurations.  A float32 field
carries about seven digits, so what is computed from one is returned in float32.
"""
import math

import numpy as np
import torch

import paper_2003_03590_gb300 as gp

TWO_PI = 2.0 * math.pi
F32_SIZES = (32, 48, 64, 96, 128, 192, 256, 512)     # lengths a float32 step is used at (and 1024)
F64_SIZES = (32, 48, 64, 96, 128, 192, 256)


def listed():
    return [
        # the smallest call: one step of a 32^3 field, where launches and latency are the time
        dict(name="step_32", kind="steps", n=32, steps=1, dt=0.004, f64=False, knk=False, minus_one=True, rings=False,
             xi_dx=1.5, tuned=False),
        # the benchmark's workload: 256^3 vortex rings, a run of steps of one tuned plan
        dict(name="steps_256", kind="steps", n=256, steps=20, dt=0.002, f64=False, knk=False, minus_one=True, rings=True,
             xi_dx=1.5, tuned=True),
        # the middle of the large grids
        dict(name="steps_512", kind="steps", n=512, steps=5, dt=0.001, f64=False, knk=False, minus_one=True, rings=False,
             xi_dx=1.5, tuned=True),
        # the largest grid (8.6 GB field), the long random-phase run of the configurations
        dict(name="steps_1024", kind="steps", n=1024, steps=2, dt=0.001, f64=False, knk=False, minus_one=True, rings=False,
             xi_dx=1.5, tuned=True),
        # the plain float64 run: ten steps, then mass and energy, as it is monitored
        dict(name="run_64_f64", kind="steps", n=64, steps=10, dt=0.005, f64=True, knk=False, minus_one=True, rings=False,
             xi_dx=2.0, tuned=False, monitor=True),
        # the float64 step as the accuracy reference of the benchmark's field, in the paper's printed order
        dict(name="steps_256_f64", kind="steps", n=256, steps=2, dt=0.002, f64=True, knk=True, minus_one=True, rings=True,
             xi_dx=1.5, tuned=False),
        # the ragged ensemble of the configurations: 24 x 64^3, 16 x 96^3, 8 x 128^3, a short run per call
        dict(name="ensemble", kind="ensemble", c64=24, c96=16, c128=8, steps=20, dt=0.004, fused=False),
        # the two gradients of an optimisation over a run: of a final-state functional with respect to the
        # initial phase, through the checkpointed steps, and of the incompressible kinetic energy
        dict(name="adjoint_128", kind="adjoint", n=128, steps=40, every=20, dt=0.002, f64=False),
        # energies, momentum, Mach numbers and spectra of the benchmark's field
        dict(name="diagnostics_256", kind="diag", n=256, f64=False),
        # the analysis of one snapshot: structure functions and helicities (a radix-3 length)
        dict(name="analysis_192", kind="analysis", n=192, order=2, f64=False),
        # imaginary-time preparation in the Taylor-Green flow with the paper's parameters
        dict(name="argle_128", kind="argle", n=128, steps=20, alpha=0.05, dtau=1.25e-2, flow="tg", renorm=False, f64=False),
        # the vortex-ring start field of the benchmark
        dict(name="rings_256", kind="rings", n=256, count=40, f64=False),
    ]


def _log_choice(rng, values):
    return values[int(rng.random() * len(values))]


def draw(rng):
    kind = _log_choice(rng, ("steps", "steps", "steps", "steps", "ensemble", "adjoint", "diag", "analysis", "argle", "rings"))
    dt = rng.choice((0.0005, 0.001, 0.002))
    if kind == "steps":
        f64 = rng.random() < 0.3
        n = _log_choice(rng, F64_SIZES if f64 else F32_SIZES)
        # a pass of at most about the points of two 1024^3 steps (float32), or two 256^3 steps (float64)
        most = max(1, min(40, (2 * 256 ** 3 if f64 else 8 * 512 ** 3) // n ** 3))
        steps = int(round(math.exp(rng.random() * math.log(most))))
        return dict(kind="steps", n=n, steps=steps, dt=dt, f64=f64, knk=rng.random() < 0.3, minus_one=rng.random() < 0.8,
                    rings=n <= 256 and rng.random() < 0.5, xi_dx=rng.choice((1.5, 2.0)), tuned=n >= 256 and rng.random() < 0.5,
                    monitor=rng.random() < 0.2)
    if kind == "ensemble":
        return dict(kind="ensemble", c64=rng.randint(1, 24), c96=rng.randint(0, 16), c128=rng.randint(0, 8),
                    steps=rng.randint(2, 20), dt=dt, fused=rng.random() < 0.5)
    if kind == "adjoint":
        every = rng.randint(3, 20)
        return dict(kind="adjoint", n=_log_choice(rng, (48, 64, 96, 128)), steps=rng.randint(1, 40), every=every, dt=dt,
                    f64=rng.random() < 0.25)
    if kind == "diag":
        return dict(kind="diag", n=_log_choice(rng, (48, 64, 96, 128, 192, 256, 512)), f64=rng.random() < 0.2)
    if kind == "analysis":
        return dict(kind="analysis", n=_log_choice(rng, (64, 96, 128, 192, 256)), order=rng.choice((2, 4, 6)), f64=False)
    if kind == "argle":
        return dict(kind="argle", n=_log_choice(rng, (48, 64, 96, 128)), steps=rng.randint(1, 20), alpha=rng.choice((0.05, 0.1)),
                    dtau=rng.choice((4e-3, 1.25e-2)), flow=rng.choice(("tg", "abc", "none")), renorm=rng.random() < 0.3,
                    f64=rng.random() < 0.2)
    return dict(kind="rings", n=_log_choice(rng, (64, 96, 128, 192, 256)), count=rng.randint(5, 40), f64=rng.random() < 0.3)


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _phase(n, seed, real, k0=None, rms=math.pi):
    """Smoothed random phase: Gaussian modes filtered by exp(-k^2 / k0^2), zero mean, scaled to the RMS."""
    k0 = k0 or (8.0 if n >= 512 else 4.0)
    m = min(n // 2 - 1, int(3 * k0))                 # modes beyond are below 1e-3 of the filter's peak
    g = _gen(seed)
    k = torch.arange(-m, m + 1, device="cuda", dtype=torch.float64)
    kx = torch.arange(0, m + 1, device="cuda", dtype=torch.float64)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kx[None, None, :] ** 2
    a = torch.randn((2 * m + 1, 2 * m + 1, m + 1, 2), generator=g, device="cuda", dtype=torch.float64)
    a = torch.view_as_complex(a) * torch.exp(-k2 / k0 ** 2)
    a[m, m, 0] = 0
    cdt = torch.complex64 if real == torch.float32 else torch.complex128
    f = torch.zeros((n, n, n // 2 + 1), device="cuda", dtype=cdt)
    idx = (torch.arange(-m, m + 1, device="cuda") % n)
    f[idx[:, None], idx[None, :], : m + 1] = a.to(cdt)
    th = torch.fft.irfftn(f, s=(n, n, n)).to(real)
    th *= rms / float(th.double().square().mean().sqrt())
    return th.contiguous()


def _xi(n, ratio):
    return ratio * TWO_PI / n


def _ring_numbers(seed, count, xi):
    r = np.random.RandomState(int(seed) % (1 << 31))
    radius = xi * (4.0 + 8.0 * r.rand(count))
    centre = TWO_PI * r.rand(count, 3)
    normal = r.randn(count, 3)
    return radius, centre, normal / np.linalg.norm(normal, axis=1)[:, None]


def _rings(n, xi, numbers, real):
    """Product of tanh-core rings with a 2 pi winding of the phase (minimum-image displacements)."""
    x = TWO_PI / n * torch.arange(n, device="cuda", dtype=real)
    psi = None
    for radius, centre, normal in zip(*numbers):
        d = [torch.remainder(x - float(c) + math.pi, TWO_PI) - math.pi for c in centre]
        d = [d[0][None, None, :], d[1][None, :, None], d[2][:, None, None]]
        zp = sum(d[j] * float(normal[j]) for j in range(3))
        rho = sum((d[j] - zp * float(normal[j])) ** 2 for j in range(3)).sqrt() - float(radius)
        s = torch.hypot(rho, zp)
        f = torch.tanh(s / (math.sqrt(2.0) * xi)) / s.clamp_min(1e-30)
        factor = torch.complex(f * rho, f * zp)
        psi = factor if psi is None else psi.mul_(factor)
    return psi.contiguous()


def _field(case, n, xi, seed):
    real = torch.float64 if case.get("f64") else torch.float32
    if case.get("rings"):
        return _rings(n, xi, _ring_numbers(seed, 40, xi), real)
    th = _phase(n, seed, real)
    return torch.polar(torch.ones_like(th), th)


def _plan_fields(case):
    prec = gp.GP_FP64 if case.get("f64") else gp.GP_FP32
    kind = case["kind"]
    if kind == "steps":
        return [gp.field_params(case["n"], case["dt"], xi_over_dx=case["xi_dx"], precision=prec,
                                split=gp.GP_SPLIT_KNK if case["knk"] else gp.GP_SPLIT_NKN, minus_one=case["minus_one"])]
    if kind == "ensemble":
        sizes = [64] * case["c64"] + [96] * case["c96"] + [128] * case["c128"]
        return [gp.field_params(n, case["dt"], xi_over_dx=1.5, precision=prec) for n in sizes]
    if kind == "argle":
        return [gp.field_params(case["n"], 0.001, alpha=case["alpha"], beta=2.0 / case["alpha"], precision=prec)]
    return [gp.field_params(case["n"], case.get("dt", 0.001), xi_over_dx=1.5, precision=prec)]


def _inputs(case, seed):
    """The tensors (and ring parameters) a pass starts from; the same for every implementation."""
    kind = case["kind"]
    if kind == "ensemble":
        sizes = [64] * case["c64"] + [96] * case["c96"] + [128] * case["c128"]
        return [_field(case, n, _xi(n, 1.5), seed * 64 + i) for i, n in enumerate(sizes)]
    n = case["n"]
    if kind == "adjoint":
        real = torch.float64 if case["f64"] else torch.float32
        cot = torch.complex(_phase(n, seed + 1, real, rms=0.7), _phase(n, seed + 2, real, rms=0.7))
        return _phase(n, seed, real), cot, _field(dict(case, rings=True), n, _xi(n, 1.5), seed)
    if kind == "rings":
        return int(seed) % (1 << 23)
    if kind == "argle":
        # a field with the flow's large scales and a non-uniform density, as during the preparation
        real = torch.float64 if case["f64"] else torch.float32
        return torch.polar(1.0 + 0.1 * torch.tanh(_phase(n, seed + 1, real)), _phase(n, seed, real, k0=3.0))
    if kind == "analysis":
        return _field(dict(case, rings=True), n, _xi(n, 1.5), seed)
    if kind == "diag":                    # a vortex tangle in a uniform flow, so that it carries momentum
        psi = _field(dict(case, rings=True), n, _xi(n, 1.5), seed)
        x = TWO_PI / n * torch.arange(n, device="cuda", dtype=torch.float64)
        ph = x[None, None, :] + 2 * x[None, :, None] - x[:, None, None]
        return psi * torch.polar(torch.ones_like(ph), ph).to(psi.dtype)
    return _field(case, n, _xi(n, case.get("xi_dx", 1.5)), seed)


FLOWS = {"none": gp.GP_FLOW_NONE, "tg": gp.GP_FLOW_TG, "abc": gp.GP_FLOW_ABC}


def prepare(case, seed):
    plan = gp.Plan(_plan_fields(case))
    if case.get("tuned"):
        plan.autotune()
    if case.get("fused"):
        plan.set_fused_batch()
    inp = _inputs(case, seed)
    if case["kind"] == "rings":
        inp = (inp, plan.empty())
    elif case["kind"] == "adjoint":
        inp[0].requires_grad_(True)
        inp[2].requires_grad_(True)
    return case, plan, inp


def _single(case, x):
    return x if case.get("f64") else np.asarray(x, dtype=np.float32)


def _spectra(case, spec):
    return {k: _single(case, v) for k, v in spec.items()}


def run(state):
    case, plan, inp = state
    kind = case["kind"]
    if kind == "steps":
        plan.step(inp, case["steps"])
        if case.get("monitor"):
            d, _ = plan.diagnostics(0, inp, spectra=False)
            return [inp, d["N"], d["E"]]
        return inp
    if kind == "ensemble":
        return plan.step(inp, case["steps"])
    if kind == "adjoint":
        theta, cot, vortices = inp
        psi = gp.GPEvolve.apply(theta, plan, case["steps"], case["every"])
        (grad,) = torch.autograd.grad(psi, theta, cot)
        J = gp.IncompressibleKineticEnergy.apply(vortices, plan, 1e-6)
        (dj,) = torch.autograd.grad(J, vortices)
        return [psi.detach(), grad, J if case["f64"] else J.float(), dj]
    if kind == "diag":
        d, spec = plan.diagnostics(0, inp)
        return [d, _spectra(case, spec)]
    if kind == "analysis":
        s = plan.structure_function(0, inp, order=case["order"])
        h, spec = plan.helicity(0, inp)
        return [_single(case, s), _single(case, [h["H"], h["H_reg"]]), _spectra(case, spec)]
    if kind == "argle":
        e = plan.argle(0, inp, FLOWS[case["flow"]], case["dtau"], case["steps"], renorm=case["renorm"])
        return [inp, e]
    seed, psi = inp
    n = case["n"]
    xi = _xi(n, 1.5)
    return plan.init_rvr(0, psi, seed, mode=0, count=case["count"], p0=4 * xi, p1=12 * xi)


# ------------------------------------------------------------------ what a pass cannot do without
def _fft_flops(n):
    return 5.0 * n ** 3 * 3 * math.log2(n)           # one complex 3D transform, radix-2 count


def work(case):
    """Each field read once and written once per step (two passes: the kinetic flow needs the whole
    field before any point of the next nonlinear flow), and the transforms' radix-2 flops."""
    kind = case["kind"]
    size = 16 if case.get("f64") else 8
    if kind == "ensemble":
        pts = [(n ** 3, n) for n, c in ((64, case["c64"]), (96, case["c96"]), (128, case["c128"])) for _ in range(c)]
        return {"bytes": float(sum(2 * size * p for p, _ in pts)),
                "flops": case["steps"] * sum(2 * _fft_flops(n) + 20 * p for p, n in pts)}
    n = case["n"]
    p = float(n) ** 3
    if kind == "steps":
        # fields within the L2 cache cross HBM once for the whole call, larger ones twice per step
        passes = 2 * case["steps"] if size * p > 60e6 else 1
        return {"bytes": passes * 2 * size * p, "flops": case["steps"] * (2 * _fft_flops(n) + 20 * p)}
    if kind == "adjoint":
        # phase, cotangent and gradient, final state, the vortex field and its gradient; the forward run, its
        # recomputation and the transposed steps; the transforms of the energy and its gradient
        return {"bytes": 5 * size * p, "flops": case["steps"] * 3 * 2 * _fft_flops(n) + 8 * _fft_flops(n)}
    if kind == "diag":
        # the three derivatives along their axes, and the transforms of the seven real fields
        return {"bytes": size * p, "flops": 2 * _fft_flops(n) + 3.5 * _fft_flops(n) + 100 * p}
    if kind == "analysis":
        ns = n // 2 + 1
        return {"bytes": size * p, "flops": 3.0 * p * ns * (1 + case["order"]) + 12 * _fft_flops(n) + 150 * p}
    if kind == "argle":
        return {"bytes": 2 * size * p, "flops": case["steps"] * (4 * _fft_flops(n) + 60 * p)}
    return {"bytes": size * p, "flops": 60.0 * case["count"] * p}


# ------------------------------------------------------------------ the same in 64 bits
def _coefficients(case, n):
    if case["kind"] == "argle":
        return case["alpha"], 2.0 / case["alpha"]
    alpha = math.sqrt(2.0) * _xi(n, case.get("xi_dx", 1.5))
    return alpha, 2.0 / alpha


def _wave(n):
    return torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64)


def _wave_d(n):
    k = _wave(n)
    if n % 2 == 0:
        k = k.clone()
        k[n // 2] = 0.0
    return k


def _k2(n):
    k = _wave(n)
    return k[None, None, :] ** 2 + k[None, :, None] ** 2 + k[:, None, None] ** 2


def _grad(psi):
    n = psi.shape[0]
    kd = _wave_d(n)
    ph = torch.fft.fftn(psi)
    return [torch.fft.ifftn(1j * k * ph) for k in (kd[None, None, :], kd[None, :, None], kd[:, None, None])]


def _nonlinear(psi, coef, shift):
    return psi * torch.exp(-1j * coef * (psi.real.square() + psi.imag.square() - shift))


def _steps(psi, alpha, beta, dt, steps, knk, minus_one):
    n = psi.shape[0]
    c = 1.0 if minus_one else 0.0
    ph = alpha * (dt / 2 if knk else dt) * _k2(n)
    K = torch.polar(torch.ones_like(ph), -ph)
    del ph
    for _ in range(steps):
        if knk:
            psi = torch.fft.ifftn(torch.fft.fftn(psi).mul_(K))
            psi = _nonlinear(psi, beta * dt, c)
            psi = torch.fft.ifftn(torch.fft.fftn(psi).mul_(K))
        else:
            psi = _nonlinear(psi, beta * dt / 2, c)
            psi = torch.fft.ifftn(torch.fft.fftn(psi).mul_(K) if not psi.requires_grad else torch.fft.fftn(psi) * K)
            psi = _nonlinear(psi, beta * dt / 2, c)
    return psi


def _mean(x):
    return float(x.mean())


def _shells(n):
    b = torch.floor(_k2(n).sqrt() + 0.5).to(torch.int64).reshape(-1)
    return b, int(math.floor(math.sqrt(3.0) * n / 2.0 + 0.5)) + 1


def _hydro(psi, alpha):
    rho = psi.real.square() + psi.imag.square()
    amp = rho.sqrt()
    ok = rho >= 1e-12
    u, q = [], []
    for g in _grad(psi):
        w = torch.conj(psi) * g
        u.append(torch.where(ok, 2 * alpha * w.imag / amp, 0.0))
        q.append(torch.where(ok, w.real / amp, 0.0))
    return rho, u, q


def _abs2(z):
    return z.real.square() + z.imag.square()


def _energy(psi, alpha, beta):
    n = psi.shape[0]
    g2 = float((_k2(n) * _abs2(torch.fft.fftn(psi))).sum()) / float(n) ** 6
    return 2 * alpha ** 2 * g2 + alpha * beta * _mean((_abs2(psi) - 1).square())


def _exact_diag(psi, alpha, beta):
    n = psi.shape[0]
    dn2 = float(n) ** 6
    rho, u, q = _hydro(psi, alpha)
    bins, nb = _shells(n)

    def binned(v):
        return torch.bincount(bins, weights=v.reshape(-1), minlength=nb)[:nb].cpu().numpy() / dn2

    e_kin = 0.5 * sum(_mean(x.square()) for x in u)
    e_q = 2 * alpha ** 2 * sum(_mean(x.square()) for x in q)
    umax = float(sum(x.square() for x in u).max())
    sq = sum(_abs2(torch.fft.fftn(x)) for x in q) * (2 * alpha ** 2)
    spec = {"E_q": binned(sq)}
    del q, sq
    kd = _wave_d(n)
    kv = (kd[None, None, :], kd[None, :, None], kd[:, None, None])
    kk = kv[0] ** 2 + kv[1] ** 2 + kv[2] ** 2
    uh = [torch.fft.fftn(x) for x in u]
    del u
    dot = sum(kv[j] * uh[j] for j in range(3)) / kk.clamp_min(1.0)
    del kk
    e_c = sum(_abs2(kv[j] * dot) for j in range(3))
    e_i = sum(_abs2(uh[j] - kv[j] * dot) for j in range(3))
    del uh, dot
    spec["E_kin_i"], spec["E_kin_c"] = 0.5 * binned(e_i), 0.5 * binned(e_c)
    del e_i, e_c
    spec["E_int"] = alpha * beta * binned(_abs2(torch.fft.fftn(rho - 1)))
    ph2 = _abs2(torch.fft.fftn(psi))
    p = [2 * alpha * float((k * ph2).sum()) / dn2 for k in kv]
    c = math.sqrt(2 * alpha * beta)
    d = {"N": _mean(rho), "E": _energy(psi, alpha, beta), "E_kin": e_kin, "E_kin_i": float(spec["E_kin_i"].sum()),
         "E_kin_c": float(spec["E_kin_c"].sum()), "E_q": e_q, "E_int": alpha * beta * _mean((rho - 1).square()),
         "P_x": p[0], "P_y": p[1], "P_z": p[2], "M_max": math.sqrt(umax) / c, "M_rms": math.sqrt(2 * e_kin) / c}
    return [d, spec]


def _exact_analysis(psi, alpha, order):
    n = psi.shape[0]
    dn = float(n) ** 3
    rho = _abs2(psi)
    g = _grad(psi)
    v = [torch.where(rho >= 1e-12, 2 * alpha * (torch.conj(psi) * x).imag / rho, 0.0) for x in g]
    s = np.zeros((3, n // 2 + 1))
    for j, (x, dim) in enumerate(zip(v, (2, 1, 0))):
        for r in range(n // 2 + 1):
            s[j, r] = _mean((torch.roll(x, -r, dims=dim) - x) ** order)
    kd = _wave_d(n)
    k = (kd[None, None, :], kd[None, :, None], kd[:, None, None])
    vh = [torch.fft.fftn(x) for x in v]
    oh = [1j * (k[1] * vh[2] - k[2] * vh[1]), 1j * (k[2] * vh[0] - k[0] * vh[2]), 1j * (k[0] * vh[1] - k[1] * vh[0])]
    om = [torch.fft.ifftn(x).real for x in oh]
    cross = [(torch.conj(g[(j + 1) % 3]) * g[(j + 2) % 3] - torch.conj(g[(j + 2) % 3]) * g[(j + 1) % 3]) for j in range(3)]
    w = [(2 * alpha / 1j * x).real for x in cross]
    ph = torch.fft.fftn(psi)
    num = torch.zeros_like(rho)
    for i in range(3):
        for j in range(3):
            num += w[i] * (torch.fft.ifftn(-k[i] * k[j] * ph) * torch.conj(g[j])).imag
    wn = sum(x.square() for x in w).sqrt()
    g2 = sum(_abs2(x) for x in g)
    keep = wn > 1e-5 * 4 * alpha * _mean(g2)
    f = torch.where(keep, 2 * alpha * num / (wn.square() * g2), 0.0)
    vr = [f * x for x in w]
    bins, nb = _shells(n)

    def spectrum(a):
        d = sum((torch.conj(a[j]) * oh[j]).real for j in range(3)).reshape(-1)
        return torch.bincount(bins, weights=d, minlength=nb)[:nb].cpu().numpy() / dn ** 2

    hs = spectrum(vh)
    h = np.array([hs.sum(), _mean(sum(vr[j] * om[j] for j in range(3)))])
    return [s, h, {"H": hs, "H_reg": spectrum([torch.fft.fftn(x) for x in vr])}]


def _flow(name, n):
    x = TWO_PI / n * torch.arange(n, device="cuda", dtype=torch.float64)
    x, y, z = x[None, None, :], x[None, :, None], x[:, None, None]
    one = torch.ones((n, n, n), device="cuda", dtype=torch.float64)
    if name == "tg":
        return [one * torch.sin(x) * torch.cos(y) * torch.cos(z), -one * torch.cos(x) * torch.sin(y) * torch.cos(z), 0 * one]
    if name == "abc":
        A, B, C = (q / math.sqrt(3.0) for q in (0.9, 1.0, 1.1))
        v = [0 * one, 0 * one, 0 * one]
        for k in (1, 2):
            v[0] += B * torch.cos(k * y) + C * torch.sin(k * z)
            v[1] += C * torch.cos(k * z) + A * torch.sin(k * x)
            v[2] += A * torch.cos(k * x) + B * torch.sin(k * y)
        return v
    return [0 * one, 0 * one, 0 * one]


def _exact_argle(psi, case):
    n, alpha, dtau = case["n"], case["alpha"], case["dtau"]
    beta = 2.0 / alpha
    v = _flow(case["flow"], n)
    v2 = sum(x.square() for x in v)
    a = dtau * alpha / 2 * _k2(n)
    target = _mean(_abs2(psi))
    for _ in range(case["steps"]):
        g = _grad(psi)
        rest = -1j * sum(v[j] * g[j] for j in range(3)) + (beta * (1 - _abs2(psi)) - v2 / (4 * alpha)) * psi
        psi = torch.fft.ifftn(((1 - a) * torch.fft.fftn(psi) + dtau * torch.fft.fftn(rest)) / (1 + a))
        if case["renorm"]:
            psi = psi * math.sqrt(target / _mean(_abs2(psi)))
    g = _grad(psi)
    e = 2 * alpha ** 2 * sum(_mean(_abs2(g[j] - 1j * v[j] / (2 * alpha) * psi)) for j in range(3))
    return [psi, e + alpha * beta * _mean((_abs2(psi) - 1).square())]


def _ekin_i(psi, alpha, eps):
    n = psi.shape[0]
    amp = (_abs2(psi) + eps).sqrt()
    u = [2 * alpha * (torch.conj(psi) * g).imag / amp for g in _grad(psi)]
    kd = _wave_d(n)
    kv = (kd[None, None, :], kd[None, :, None], kd[:, None, None])
    kk = (kv[0] ** 2 + kv[1] ** 2 + kv[2] ** 2).clamp_min(1.0)
    uh = [torch.fft.fftn(x) for x in u]
    dot = sum(kv[j] * uh[j] for j in range(3)) / kk
    return 0.5 * sum(_abs2(uh[j] - kv[j] * dot).sum() for j in range(3)) / float(n) ** 6


_GAMMA, _M64 = 0x9E3779B97F4A7C15, (1 << 64) - 1


def _splitmix(c):
    z = ((c + 1) * _GAMMA) & _M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def _documented_rings(seed, count, xi):
    """The ring parameters of the documented stream: positions seed 2^40 + 8 j + c."""
    radius, centre, normal = [], [], []
    for j in range(count):
        v = [_splitmix((seed << 40) + 8 * j + c) for c in range(8)]
        u = [(q >> 11) * 2.0 ** -53 for q in v]
        radius.append(4 * xi + 8 * xi * u[0])
        centre.append([TWO_PI * q for q in u[1:4]])
        r0 = math.sqrt(-2.0 * math.log(((v[4] >> 11) + 1) * 2.0 ** -53))
        r1 = math.sqrt(-2.0 * math.log(((v[6] >> 11) + 1) * 2.0 ** -53))
        t0, t1 = TWO_PI * u[5], TWO_PI * u[7]
        m = [r0 * math.cos(t0), r0 * math.sin(t0), r1 * math.cos(t1)]
        s = math.sqrt(sum(q * q for q in m))
        normal.append([q / s for q in m])
    return radius, centre, normal


def exact(case, seed):
    kind = case["kind"]
    if kind == "steps" and case["n"] > 512:
        return None                       # several 17 GB arrays per operation: over the time allowed
    inp = _inputs(case, seed)
    if kind == "rings":
        xi = _xi(case["n"], 1.5)
        return _rings(case["n"], xi, _documented_rings(inp, case["count"], xi), torch.float64)
    if kind == "ensemble":
        out = []
        for f in inp:
            alpha, beta = _coefficients(case, f.shape[0])
            out.append(_steps(f.to(torch.complex128), alpha, beta, case["dt"], case["steps"], False, True))
        return out
    alpha, beta = _coefficients(case, case["n"])
    if kind == "adjoint":
        th = inp[0].double().requires_grad_(True)
        psi = torch.polar(torch.ones_like(th), th)
        psi = _steps(psi, alpha, beta, case["dt"], case["steps"], False, True)
        (grad,) = torch.autograd.grad(psi, th, inp[1].to(torch.complex128))
        vortices = inp[2].to(torch.complex128).requires_grad_(True)
        J = _ekin_i(vortices, alpha, 1e-6)
        (dj,) = torch.autograd.grad(J, vortices)
        return [psi.detach(), grad, J.detach(), dj]
    psi = inp.to(torch.complex128)
    if kind == "steps":
        psi = _steps(psi, alpha, beta, case["dt"], case["steps"], case["knk"], case["minus_one"])
        return [psi, _mean(_abs2(psi)), _energy(psi, alpha, beta)] if case.get("monitor") else psi
    if kind == "diag":
        return _exact_diag(psi, alpha, beta)
    if kind == "analysis":
        return _exact_analysis(psi, alpha, case["order"])
    return _exact_argle(psi, case)
