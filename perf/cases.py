"""The calls whose time is measured: convolutions A_n u (paper Sec. 2.1) and Lippmann-Schwinger
solves (Sec. 3.3) through the package's public entry points, from one 64 x 64 density to batches of
4096 x 4096, in FP64 and FP32, with each transform grid, output type and call form in use.

    listed()             the cases;  draw(rng): one more of the same ranges
    prepare(case, seed)  plans and inputs, on the GPU
    run(state)           one call, its whole outputs
    work(case)           bytes and flops the call cannot do without
    exact(case, seed)    the same outputs in 64-bit torch, without the package

A case's "call" is the entry point: "apply" (ConvPlan.apply), "multi" (apply_multi: five kernels on
the same densities), "group" (ConvGroup: mixed sizes in one graph launch), "ls" (ls_solve on a plan
that the program keeps), "ls_fresh" (a plan built for the request, solved with, and closed: what a
served solve with a new wavenumber does).
"""
import math

import numpy as np
import torch

from paper_2107_03958_gb300.api import ConvGroup, ConvPlan, apply_multi, ls_solve

LAPLACE = -1.0 / (2.0 * math.pi)
SWEEP = (("log", 0.0, 0.0), ("pow", -0.5, 0.0), ("pow", -1.0, 0.0), ("pow", -1.5, 0.0), ("helmholtz", 0.0, 20.0))
GROUP_SIZES = (128, 256, 512, 1024, 2048)


def _conv(name, kernel, n, batch, precision, gamma=0.0, kappa=0.0, grid="compact", mask=False, call="apply"):
    c = {"call": call, "kernel": kernel, "gamma": gamma, "kappa": kappa, "n": n, "batch": batch,
         "precision": precision, "grid": grid, "mask": mask}
    return dict(c, name=name) if name else c


def _group(name, base, kernel_shift, precision):
    c = {"call": "group", "base": base, "shift": kernel_shift, "precision": precision}
    return dict(c, name=name) if name else c


def _ls(name, n, kappa, precision, contrast="bump", call="ls"):
    c = {"call": call, "n": n, "kappa": kappa, "precision": precision, "contrast": contrast}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small density, the plain method on the period-2 grid (64 x 64, a = 1.1): latency and launches
        _conv("bump_fp64_n64", "log", 64, 1, "fp64", grid="period2"),
        # the kernel sweep's three sizes in FP64, batch 16: a real kernel at 256, the complex
        # Helmholtz kernel at 1024, the largest batch at 4096
        _conv("sweep_fp64_n256_b16", "pow", 256, 16, "fp64", gamma=-0.5),
        _conv("helm_fp64_n1024_b16", "helmholtz", 1024, 16, "fp64", kappa=20.0),
        _conv("sweep_fp64_n4096_b16", "log", 4096, 16, "fp64"),
        # discontinuous densities with the Fourier-smoothing mask on the paper's period-3 grid, at a
        # size of the paper's timing series n = 24 l (not a power of two)
        _conv("disc_fs_fp64_n480_b8", "pow", 480, 8, "fp64", gamma=-1.0, grid="period3", mask=True),
        # a server's mixed-size batch of small and middling convolutions in one graph launch
        _group("mix_fp32_group", 16, 0, "fp32"),
        # the FP32 sweep at its largest size
        _conv("sweep_fp32_n4096_b16", "pow", 4096, 16, "fp32", gamma=-1.0),
        # the paper's tables: several kernels applied to the same densities
        _conv("multi_fp32_n2048_b4", "sweep", 2048, 4, "fp32", call="multi"),
        # FP32 on the paper's own period-3 grid with the complex kernel
        _conv("helm_fp32_p3_n1024_b16", "helmholtz", 1024, 16, "fp32", kappa=20.0, grid="period3"),
        # Lippmann-Schwinger: all-FP64, and FP32 matvecs with FP64 refinement
        _ls("ls_fp64_n512_k40", 512, 40.0, "fp64"),
        _ls("ls_mixed_n1024_k40", 1024, 40.0, "mixed"),
        # a served solve: its wavenumber is new, so its plan is built on the request's path
        _ls("ls_fresh_mixed_n256_k33", 256, 33.0, "mixed", call="ls_fresh"),
    ]


def _smooth_sizes(lo, hi, even):
    return [n for n in range(lo, hi + 1) if _is_smooth(n) and not (even and n % 2)]


def _is_smooth(n):
    for f in (2, 3, 5):
        while n % f == 0:
            n //= f
    return n == 1


def _log_pick(rng, sizes):
    """A size near a log-uniform point of the range, so that small and large ones are drawn alike."""
    t = math.exp(rng.uniform(math.log(sizes[0]), math.log(sizes[-1])))
    return min(sizes, key=lambda n: abs(math.log(n / t)))


def draw(rng):
    kind = rng.choice(["conv64", "conv64", "conv64", "conv32", "conv32", "conv32", "multi", "group", "ls", "ls", "ls_fresh"])
    kappa = round(rng.uniform(5.0, 60.0), 2)
    if kind in ("ls", "ls_fresh"):
        n = rng.choice([128, 256, 512, 1024] if kind == "ls" else [128, 256, 512])
        return _ls(None, n, kappa, rng.choice(["fp64", "mixed"]), rng.choice(["bump", "disk"]), call=kind)
    if kind == "group":
        return _group(None, rng.randint(2, 20), rng.randint(0, 4), rng.choice(["fp32", "fp64"]))
    precision = "fp64" if kind == "conv64" or (kind == "multi" and rng.random() < 0.5) else "fp32"
    if kind == "multi":
        n = rng.choice([64, 128, 256, 512, 1024, 2048])
        return _conv(None, "sweep", n, rng.randint(1, 4), precision, call="multi")
    grid = rng.choice(["compact", "compact", "compact", "period3", "period2"])
    # powers of two are what sweeps, servers and solves use; the rest are the paper's n = 24 l and odd sizes
    pow2 = rng.random() < 0.6
    top = {"compact": 4096, "period3": 2048, "period2": 1024}[grid]
    if pow2:
        n = _log_pick(rng, [64 << i for i in range(7) if 64 << i <= top])
    else:
        n = _log_pick(rng, _smooth_sizes(48, min(top, 1280), even=grid != "period2"))
    # at most a quarter of the largest listed case's points where the grid or the size is less regular
    cap = 16 * 4096 * 4096 // (4 if precision == "fp64" or not pow2 or grid != "compact" else 1)
    batch = max(1, min(rng.choice([1, 2, 3, 5, 8, 11, 16]), cap // (n * n)))
    kernel, gamma, kap = rng.choice([("log", 0.0, 0.0), ("pow", rng.choice([-0.5, -1.0, -1.5]), 0.0),
                                     ("helmholtz", 0.0, kappa), ("yukawa", 0.0, kappa)])
    return _conv(None, kernel, n, batch, precision, gamma, kap, grid, mask=rng.random() < 0.25)


# ------------------------------------------------------------------------------------ inputs
def _axis(n):
    return torch.arange(n, dtype=torch.float64, device="cuda") / n


def _add_bump(out, c1, c2, r, amp):
    """out += amp exp(-1 / (1 - |x - c|^2 / r^2)) inside the disk of radius r."""
    n = out.shape[-1]
    x = _axis(n)
    i0, i1 = max(0, int((c1 - r) * n)), min(n, int((c1 + r) * n) + 2)
    j0, j1 = max(0, int((c2 - r) * n)), min(n, int((c2 + r) * n) + 2)
    t = ((x[i0:i1, None] - c1) ** 2 + (x[None, j0:j1] - c2) ** 2) / (r * r)
    out[i0:i1, j0:j1] += torch.where(t < 1.0, amp * torch.exp(-1.0 / torch.clamp(1.0 - t, min=1e-300)), 0.0)


def _densities(n, batch, rng, dtype):
    """Sums of one to eight smooth bumps: centres in [0.2, 0.8]^2, radii in [0.05, 0.2], normal amplitudes."""
    u = torch.zeros((batch, n, n), dtype=dtype, device="cuda")
    for b in range(batch):
        d = torch.zeros((n, n), dtype=torch.float64, device="cuda")
        for _ in range(int(rng.integers(1, 9))):
            c = rng.uniform(0.2, 0.8, 2)
            _add_bump(d, float(c[0]), float(c[1]), float(rng.uniform(0.05, 0.2)), float(rng.standard_normal()))
        u[b] = d
    return u


def _smoothed_disk(n, rng, dtype):
    """A seeded indicator-like mask: a disk with a narrow smooth rim (the mask multiplies the density)."""
    c = rng.uniform(0.45, 0.55, 2)
    x = _axis(n)
    r = torch.sqrt((x[:, None] - float(c[0])) ** 2 + (x[None, :] - float(c[1])) ** 2)
    return (0.5 * torch.erfc((r - 0.3) * 40.0)).to(dtype)


def _conv_inputs(case, seed):
    rng = np.random.default_rng([seed, case["n"], case["batch"]])
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    u = _densities(case["n"], case["batch"], rng, dtype)
    return u, (_smoothed_disk(case["n"], rng, dtype) if case["mask"] else None)


def _group_items(case):
    """(n, batch, kernel, gamma, kappa) of each item: fewer densities the larger the grid."""
    return [(n, max(1, case["base"] * 128 // n), *SWEEP[(i + case["shift"]) % 5]) for i, n in enumerate(GROUP_SIZES)]


def _group_inputs(case, seed):
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    return [_densities(n, b, np.random.default_rng([seed, n, b]), dtype) for n, b, *_ in _group_items(case)]


def _ls_inputs(case, seed):
    """The contrast (a smooth bump or a disk, 0.5 high) and a plane wave from a seeded direction."""
    rng = np.random.default_rng([seed, case["n"]])
    n, x = case["n"], _axis(case["n"])
    c = rng.uniform(0.47, 0.53, 2)
    m = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    if case["contrast"] == "bump":
        _add_bump(m, float(c[0]), float(c[1]), 0.4, 0.5)
    else:
        r2 = (x[:, None] - float(c[0])) ** 2 + (x[None, :] - float(c[1])) ** 2
        m += 0.5 * (r2 < 0.09)
    th = float(rng.uniform(0.0, 2.0 * math.pi))
    ph = case["kappa"] * (x[:, None] * math.cos(th) + x[None, :] * math.sin(th))
    return m, torch.complex(torch.cos(ph), torch.sin(ph))


# ------------------------------------------------------------------------------------ the calls
def _plan(kernel, gamma, kappa, n, batch, precision, grid):
    return ConvPlan(kernel, n=n, period=2 if grid == "period2" else 3, trunc_a=1.1 if grid == "period2" else 0.0,
                    precision=precision, io="r2c" if kernel == "helmholtz" else "r2r", batch_max=batch, gamma=gamma,
                    kappa=kappa, scale=LAPLACE if kernel == "log" else 1.0, compact=grid == "compact")


def _ls_plan(case):
    return ConvPlan("helmholtz", n=case["n"], period=3, precision="fp32" if case["precision"] == "mixed" else "fp64",
                    io="c2c", kappa=case["kappa"], compact=True)


def prepare(case, seed):
    call = case["call"]
    if call in ("ls", "ls_fresh"):
        m, f = _ls_inputs(case, seed)
        return {"case": case, "m": m, "f": f, "plan": _ls_plan(case) if call == "ls" else None}
    if call == "group":
        items = []
        for (n, b, kernel, gamma, kappa), u in zip(_group_items(case), _group_inputs(case, seed)):
            p = _plan(kernel, gamma, kappa, n, b, case["precision"], "compact")
            items.append((p, u, torch.empty(u.shape, dtype=p.out_dtype(), device="cuda")))
        return {"case": case, "group": ConvGroup(items), "outs": [it[2] for it in items]}
    u, mask = _conv_inputs(case, seed)
    if call == "multi":
        plans = [_plan(k, g, kap, case["n"], case["batch"], case["precision"], case["grid"]) for k, g, kap in SWEEP]
        return {"case": case, "plans": plans, "u": u, "mask": mask}
    p = _plan(case["kernel"], case["gamma"], case["kappa"], case["n"], case["batch"], case["precision"], case["grid"])
    return {"case": case, "plan": p, "u": u, "mask": mask}


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "apply":
        return state["plan"].apply(state["u"], mask=state["mask"])
    if call == "multi":
        return apply_multi(state["plans"], state["u"], mask=state["mask"])
    if call == "group":
        state["group"].launch()
        return state["outs"]
    plan = state["plan"] if call == "ls" else _ls_plan(case)
    x, _ = ls_solve(plan, state["m"], state["f"], tol=1e-10, refine=case["precision"] == "mixed")
    if call == "ls_fresh":
        plan.close()
    return x


# ------------------------------------------------------------------------------------ work
def _conv_work(kernel, n, batch, e):
    """One batch on the 2n-periodic grid, the smallest that holds the linear convolution: the density
    read, the result written, the multiplier's quadrant read; the flops of the zero-padded real
    transform forward and the cropped one (real or complex) back."""
    cplx = kernel == "helmholtz"
    points = 4.0 * n * n
    flops = batch * 0.75 * (2.5 + (5.0 if cplx else 2.5)) * points * math.log2(points)
    return batch * n * n * e * (3 if cplx else 2) + (n + 1) ** 2 * e * (2 if cplx else 1), flops


def work(case):
    call = case["call"]
    if call in ("ls", "ls_fresh"):
        # GMRES steps to 1e-10 grow with the wavenumber (about 8 at 10, 14 at 40); each needs one
        # complex convolution and reads its vector; the contrast, field and solution move once
        n, steps = case["n"], 6.0 + 0.2 * case["kappa"]
        points = 4.0 * n * n
        return {"bytes": n * n * (8 + 16 + 16) + steps * n * n * 32, "flops": steps * 7.5 * points * math.log2(points)}
    e = 8 if case["precision"] == "fp64" else 4
    if call == "group":
        parts = [_conv_work(it[2], it[0], it[1], e) for it in _group_items(case)]
    elif call == "multi":
        parts = [_conv_work(k, case["n"], case["batch"], e) for k, _, _ in SWEEP]
        parts.append((-4 * case["batch"] * case["n"] ** 2 * e, 0.0))  # the densities are read once
    else:
        parts = [_conv_work(case["kernel"], case["n"], case["batch"], e)]
        if case["mask"]:
            parts.append((case["n"] ** 2 * e, 0.0))
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ------------------------------------------------------------------------------------ exact
def _hankel(order, x):
    """P, Q of Hankel's expansion J = sqrt(2 / (pi x)) (P cos(chi) - Q sin(chi)), for x >= 25."""
    p, q, c = torch.ones_like(x), torch.zeros_like(x), torch.ones_like(x)
    for k in range(1, 24):
        c = c * ((4 * order * order - (2 * k - 1) ** 2) / (8.0 * k)) / x
        if k % 2:
            q = q + (c if k % 4 == 1 else -c)
        else:
            p = p + (c if k % 4 == 0 else -c)
    return p, q


def _j(order, x):
    """J0 or J1: the trapezoidal rule for Bessel's integral (exponentially accurate) below 25, Hankel's
    expansion beyond."""
    v = torch.empty_like(x)
    near = x < 25.0
    xn = x[near]
    if xn.numel():
        acc = torch.zeros_like(xn)
        for i in range(64):
            th = 2.0 * math.pi * (i + 0.5) / 64
            acc += torch.cos(order * th - xn * math.sin(th))
        v[near] = acc / 64
    xf = x[~near]
    if xf.numel():
        p, q = _hankel(order, xf)
        # cos and sin of x - pi/4 - order pi/2 from those of x (no rounded subtraction)
        co, si = torch.cos(xf), torch.sin(xf)
        cc, ss = ((co + si), (si - co)) if order == 0 else ((si - co), -(si + co))
        v[~near] = torch.sqrt(1.0 / (math.pi * xf)) * (p * cc - q * ss)
    return v


def _y0(x):
    """Y0: the logarithmic series below 6, the integral over (0, pi) and the decaying one beyond."""
    v = torch.empty_like(x)
    near = x < 6.0
    t = 0.25 * x[near] ** 2
    acc, term, harmonic = torch.zeros_like(t), torch.ones_like(t), 0.0
    for k in range(1, 40):
        term = -term * t / (k * k)
        harmonic += 1.0 / k
        acc = acc - term * harmonic
    v[near] = (2.0 / math.pi) * ((torch.log(0.5 * x[near]) + 0.57721566490153286061) * _j(0, x[near]) + acc)
    v[~near] = _y_integral(0, x[~near])
    return v


def _y_integral(order, x):
    t, w = _gauss(400)
    x = x[..., None]
    th = math.pi * t
    first = (w * torch.sin(x * torch.sin(th) - order * th)).sum(-1)
    top = math.asinh(45.0 / 5.0)  # exp(-x sinh t) is below 1e-19 there for x >= 5
    sh, ex = torch.sinh(top * t), torch.exp(top * t)
    grow = 2.0 if order == 0 else ex - 1.0 / ex
    return first - (top / math.pi) * (w * grow * torch.exp(-x * sh)).sum(-1)


def _k01(x):
    """K0 and K1 by the trapezoidal rule for the integral of exp(-x cosh t) cosh(order t)."""
    t = np.arange(0, 4000) * 0.0025
    f = np.exp(-x * np.cosh(t)) * 0.0025
    f[0] *= 0.5
    return float(f.sum()), float((f * np.cosh(t)).sum())


def _gauss(count):
    t, w = np.polynomial.legendre.leggauss(count)
    return torch.tensor(0.5 * (t + 1.0), device="cuda"), torch.tensor(0.5 * w, device="cuda")


def _pow_moments(s, a, gamma):
    """int_0^a rho^(1+gamma) J0(s rho) d rho: Gauss rule in t (rho = a t^2) to z = s a = 60, beyond it
    the constant of the half-line integral minus its tail by repeated integration by parts."""
    z = s * a
    v = torch.zeros_like(s)
    near = z <= 60.0
    t, w = _gauss(240)
    zn = z[near]
    f = w * t ** (3.0 + 2.0 * gamma)
    v[near] = 2.0 * a ** (2.0 + gamma) * (f * _j(0, zn[:, None] * t * t)).sum(1)
    far = ~near
    zf, sf = z[far], s[far]
    nu = 1.0 + gamma
    c, p, q = torch.ones_like(zf), torch.zeros_like(zf), torch.zeros_like(zf)
    for k in range(12):
        p = p + c
        q = q + c * (nu - 1.0 - 2.0 * k)
        c = -c * (nu - 1.0 - 2.0 * k) ** 2 / (zf * zf)
    half_line = 2.0 ** nu * math.gamma(1.0 + 0.5 * gamma) / math.gamma(-0.5 * gamma)
    v[far] = sf ** (-1.0 - nu) * (half_line + _j(1, zf) * zf ** nu * p + _j(0, zf) * zf ** (nu - 1.0) * q)
    return v


def _helmholtz_moments(s, a, kappa):
    """(i/4) H0(kappa r): the closed form, and a Gauss rule (rho = a u^4) where s is near kappa."""
    ka = torch.tensor([kappa * a], dtype=torch.float64, device="cuda")
    H0 = torch.complex(_j(0, ka), _y0(ka))
    H1 = torch.complex(_j(1, ka), _y_integral(1, ka))
    z = s * a
    band = (s - kappa).abs() < 0.1 * kappa
    d = torch.where(band, torch.ones_like(s), s * s - kappa * kappa)
    g = 0.5j * math.pi * (z * _j(1, z) * H0 - ka * _j(0, z) * H1 - 2j / math.pi) / d
    u, w = _gauss(600)
    r = a * u ** 4
    f = w * 4.0 * a * u ** 3 * r * torch.complex(_j(0, kappa * r), _y0(kappa * r))
    g[band] = 0.5j * math.pi * (f * _j(0, s[band][:, None] * r)).sum(1)
    return g


def _moments(kernel, gamma, kappa, M, b, a):
    """The multiplier on the M x M frequency grid (FFT order), 2 pi int_0^a g(rho) J0(s rho) rho d rho,
    evaluated for 0 <= k1, k2 <= M/2; _convolve mirrors it.  The log kernel is -log|x| / (2 pi)."""
    k = torch.arange(M // 2 + 1, dtype=torch.float64, device="cuda")
    s = (2.0 * math.pi / b) * torch.sqrt(k[:, None] ** 2 + k[None, :] ** 2)
    z = s * a
    if kernel == "log":
        g = -a * math.log(a) * _j(1, z) / s + (1.0 - _j(0, z)) / (s * s)
        g[0, 0] = 0.25 * a * a * (1.0 - 2.0 * math.log(a))
    elif kernel == "pow":
        g = 2.0 * math.pi * _pow_moments(s.flatten(), a, gamma).reshape(s.shape)
    elif kernel == "yukawa":
        ka = kappa * a
        K0, K1 = _k01(ka)
        g = (1.0 + z * _j(1, z) * K0 - ka * _j(0, z) * K1) / (s * s + kappa * kappa)
    else:
        g = _helmholtz_moments(s.flatten(), a, kappa).reshape(s.shape)
    return g


def _convolve(u, g, M):
    """A_n u = crop(ifft2(g fft2(u extended by zeros))) for one n x n density, rows and columns apart."""
    n = u.shape[0]
    idx = torch.arange(M, device="cuda")
    idx = torch.minimum(idx, M - idx)
    real = not (u.is_complex() or g.is_complex())
    w = torch.fft.fft(u.to(torch.complex128), n=M, dim=1)
    cols = M // 2 + 1 if real else M
    for c in range(0, cols, 1024):  # columns in chunks: bounded memory
        e = min(cols, c + 1024)
        v = torch.fft.fft(w[:, c:e], n=M, dim=0)
        v *= g[idx[:, None], idx[c:e]]
        w[:, c:e] = torch.fft.ifft(v, dim=0)[:n]
    return torch.fft.irfft(w[:, :cols], n=M, dim=1)[:, :n] if real else torch.fft.ifft(w, dim=1)[:, :n]


def _grid_of(case_grid, n):
    b = 2.0 if case_grid == "period2" else 3.0
    return int(round(b * n)), b, 1.1 if case_grid == "period2" else 0.5 * (math.sqrt(2.0) + 2.0)


def _exact_conv(u, mask, kernel, gamma, kappa, grid):
    M, b, a = _grid_of(grid, u.shape[-1])
    g = _moments(kernel, gamma, kappa, M, b, a)
    m = 1.0 if mask is None else mask.double()
    return torch.stack([_convolve(d.double() * m, g, M) for d in u])


def _exact_solve(case, seed):
    """u + kappa^2 A_n(m u) = f by GMRES to 1e-14 in complex128."""
    m, f = _ls_inputs(case, seed)
    M, b, a = _grid_of("period3", case["n"])
    g = _moments("helmholtz", 0.0, case["kappa"], M, b, a)
    k2 = case["kappa"] ** 2

    def op(v):
        return v + k2 * _convolve(m * v, g, M)

    x = torch.zeros_like(f)
    for _ in range(3):
        r = f - op(x)
        beta = float(torch.linalg.vector_norm(r))
        if beta <= 1e-14 * float(torch.linalg.vector_norm(f)):
            break
        V, H = [r / beta], np.zeros((61, 60), dtype=complex)
        for j in range(60):
            w = op(V[j])
            for _again in range(2):
                for i in range(j + 1):
                    c = complex(torch.vdot(V[i].flatten(), w.flatten()))
                    H[i, j] += c
                    w = w - c * V[i]
            H[j + 1, j] = float(torch.linalg.vector_norm(w))
            V.append(w / H[j + 1, j].real)
            e = np.zeros(j + 2, dtype=complex)
            e[0] = beta
            y, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
            if np.linalg.norm(H[:j + 2, :j + 1] @ y - e) <= 1e-13 * beta:
                break
        for i, c in enumerate(y):
            x = x + complex(c) * V[i]
    return x


def exact(case, seed):
    call = case["call"]
    if call in ("ls", "ls_fresh"):
        return _exact_solve(case, seed)
    if call == "group":
        return [_exact_conv(u, None, k, g, kap, "compact")
                for (n, b, k, g, kap), u in zip(_group_items(case), _group_inputs(case, seed))]
    u, mask = _conv_inputs(case, seed)
    if call == "multi":
        return [_exact_conv(u, mask, k, g, kap, case["grid"]) for k, g, kap in SWEEP]
    return _exact_conv(u, mask, case["kernel"], case["gamma"], case["kappa"], case["grid"])
