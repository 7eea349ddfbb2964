"""Cases for timing the solver through its public entry points.

Each case is one call, or one short chain of calls, of a program that models or inverts
microseismic wavefields with this package: operator applications of every precision, the adjoint
and the gradients of an inversion, the work a new frequency costs, a batched mixed-precision solve
and a differentiable forward + backward step.  Media, fields and sources are synthetic, made on the
GPU from the seed; their values follow the models the solver is used on (a 3000 m/s background with
a few per cent of smooth anisotropic contrast, wavefields a few nodes per wavelength).

``exact`` evaluates the same quantities with plain torch in complex128 (dense FFT convolution,
autograd for the adjoint and the gradients), without the package.
"""
import math

import numpy as np
import torch

from paper_2301_12836_gb300 import autograd, lsm

VP, VS, RHO = 3000.0, 1730.0, 2300.0
MU = RHO * VS * VS
LAM = RHO * VP * VP - 2.0 * MU
_PAIRS = [(i, j) for i in range(6) for j in range(i, 6)]
_ORTHO = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2), (3, 3), (4, 4), (5, 5)]
_OPS = ("apply_f64", "apply_f32", "apply_df", "adjoint", "gradient", "frequency", "solve", "receivers")
# nodes of the largest grid a drawn case may have, and of the smallest
_RANGE = {"apply_f64": (16 ** 3, 128 ** 3), "apply_f32": (48 ** 3, 200 ** 3), "apply_df": (32 ** 3, 128 ** 3),
          "adjoint": (24 ** 3, 110 ** 3), "gradient": (24 ** 3, 110 ** 3), "frequency": (24 ** 3, 110 ** 3),
          "solve": (24 ** 3, 100 ** 3), "receivers": (12 ** 3, 40 ** 3)}


def _case(name, op, n, dx, freq, medium, nsrc=1):
    return {"name": name, "op": op, "nx": n[0], "ny": n[1], "nz": n[2], "dx": dx, "freq": freq, "medium": medium,
            "nsrc": nsrc}


def listed():
    return [
        # the smallest model of the tests (a VTI cube in a 16^3 grid): one FP64 operator application
        # of a user's own iteration, where launches and latency are all the time
        _case("apply_f64_16", "apply_f64", (16, 16, 16), 10.0, 10.0, "inclusion"),
        # a survey box whose sides are not powers of two, no two alike, one of them odd
        _case("apply_f64_ragged", "apply_f64", (60, 45, 50), 10.0, 12.0, "full"),
        # the operator in double precision at the size of the batched benchmark: the refinement
        # residual of a mixed solve, or one half step of a plain FP64 BiCGSTAB
        _case("apply_f64_128", "apply_f64", (128, 128, 128), 8.0, 20.0, "ortho"),
        # the single-precision operator of an inner iteration on the three-layer model's grid, one
        # system at a time: an ordinary call that does not fill the GPU by itself
        _case("apply_f32_64", "apply_f32", (64, 64, 64), 10.0, 15.0, "layers"),
        # the same at the size of the batched benchmark
        _case("apply_f32_128", "apply_f32", (128, 128, 128), 8.0, 20.0, "ortho"),
        # the largest grid the library takes: a 1.3 km fractured (tilted TI) reservoir box
        _case("apply_f32_256", "apply_f32", (256, 256, 256), 5.0, 30.0, "full"),
        # the double-float operator: the refinement residual of handles that ask for it
        _case("apply_df_128", "apply_df", (128, 128, 128), 8.0, 20.0, "ortho"),
        # inversion on the layered 96^3 model: one application of the adjoint operator ...
        _case("adjoint_96", "adjoint", (96, 96, 96), 10.0, 16.0, "layers"),
        # ... and the contrast and moment-tensor gradients from a forward and an adjoint field
        _case("gradient_96", "gradient", (96, 96, 96), 10.0, 16.0, "layers"),
        # what every new frequency of a sweep costs before its solves: the Green spectrum, the
        # background fields of eight moment tensors, and a first residual
        _case("frequency_128", "frequency", (128, 128, 128), 8.0, 24.0, "ortho", 8),
        # the batched mixed-precision solve, eight sources of one frequency, to the library's
        # default tolerance
        _case("solve_mixed_128x8", "solve", (128, 128, 128), 8.0, 10.0, "ortho", 8),
        # one step of an inversion: receiver data of two frequencies and its gradients
        _case("receivers_f64_32", "receivers", (32, 32, 32), 10.0, 8.0, "layers", 2),
    ]


def _side(rng, lo, hi):
    """A side between lo and hi (log-uniform) whose double has no prime factor above 5."""
    ok = [n for n in range(max(4, lo), hi + 1) if _smooth(n)]
    t = math.exp(rng.uniform(math.log(ok[0]), math.log(ok[-1])))
    return min(ok, key=lambda n: abs(math.log(n / t)))


def _smooth(n):
    for p in (2, 3, 5):
        while n % p == 0:
            n //= p
    return n == 1


def draw(rng):
    op = rng.choice(_OPS)
    lo, hi = _RANGE[op]
    nodes = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    side = nodes ** (1.0 / 3.0)
    if rng.random() < 0.25:   # a cube whose side is a power of two, as users like them
        s = max(8, min(128, 2 ** round(math.log2(side))))
        n = (s, s, s)
    else:
        n = tuple(min(200, _side(rng, int(0.6 * side), int(1.5 * side) + 1)) for _ in range(3))
        while n[0] * n[1] * n[2] > hi:
            n = tuple(_side(rng, 4, max(4, int(0.9 * v))) for v in n)
    dx = rng.choice([5.0, 8.0, 10.0])
    # 10 to 30 nodes of the grid per shear wavelength; whole solves at the low end of the frequencies,
    # where the iteration converges on every medium here
    nodes_per_wave = rng.uniform(10.0, 30.0) if op not in ("solve", "receivers") else rng.uniform(24.0, 40.0)
    medium = rng.choice(["inclusion", "ortho", "full", "layers"]) if op not in ("solve", "receivers") else rng.choice(["inclusion", "ortho", "layers"])
    nsrc = rng.choice([1, 2, 3, 4, 6, 8]) if op in ("frequency", "solve") else (rng.choice([1, 2, 3]) if op == "receivers" else 1)
    c = _case("", op, n, dx, round(VS / (dx * nodes_per_wave), 2), medium, nsrc)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _smooth_noise(shape, gen, corr):
    """Zero-mean unit-std real field with a Gaussian covariance of `corr` nodes."""
    w = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    ks = [torch.fft.fftfreq(s, device="cuda", dtype=torch.float64) * (2.0 * math.pi) for s in shape[:-1]]
    ks.append(torch.fft.rfftfreq(shape[-1], device="cuda", dtype=torch.float64) * (2.0 * math.pi))
    k2 = ks[0][:, None, None] ** 2 + ks[1][None, :, None] ** 2 + ks[2][None, None, :] ** 2
    f = torch.fft.irfftn(torch.fft.rfftn(w) * torch.exp(-k2 * (corr * corr / 8.0)), s=shape)
    f -= f.mean()
    return f / f.std()


def _wavefield(n, gen):
    """Three smooth complex components (about ten nodes per wavelength) with 5% of white noise."""
    shape = (n[2], n[1], n[0])
    out = torch.empty((3,) + shape, device="cuda", dtype=torch.complex128)
    for c in range(3):
        for part in ("real", "imag"):
            f = _smooth_noise(shape, gen, 3.0)
            f += 0.05 * torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
            getattr(out[c], part).copy_(f)
    return out


def _vti(vp, vs, eps, delta, gamma):
    c33, c44 = RHO * vp * vp, RHO * vs * vs
    c11, c66 = c33 * (1.0 + 2.0 * eps), c44 * (1.0 + 2.0 * gamma)
    c13 = math.sqrt(2.0 * delta * c33 * (c33 - c44) + (c33 - c44) ** 2) - c44
    C = np.zeros((6, 6))
    C[0, 0] = C[1, 1] = c11
    C[2, 2] = c33
    C[0, 1] = C[1, 0] = c11 - 2.0 * c66
    C[0, 2] = C[2, 0] = C[1, 2] = C[2, 1] = c13
    C[3, 3] = C[4, 4] = c44
    C[5, 5] = c66
    return C


def _medium(case, gen, rs):
    """Contrast (21 planes) and density contrast of the case's medium."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape = (nz, ny, nx)
    iso = _vti(VP, VS, 0.0, 0.0, 0.0)
    dC = torch.zeros((21,) + shape, device="cuda", dtype=torch.float64)
    drho = torch.zeros(shape, device="cuda", dtype=torch.float64)
    kind = case["medium"]
    if kind == "inclusion":      # a VTI block in the middle of an isotropic box
        C = _vti(VP, VS, *rs.uniform(0.04, 0.12, 3)) - iso
        sl = tuple(slice(max(1, (5 * s) // 16), max(2, (11 * s) // 16)) for s in shape)
        for k, (i, j) in enumerate(_PAIRS):
            dC[(k,) + sl] = C[i, j]
        drho[sl] = 0.05 * RHO
    elif kind == "layers":       # three horizontal VTI layers with a 2% smooth perturbation
        b = [0, (nz + 1) // 3, (2 * nz + 1) // 3, nz]
        for m, v in enumerate((0.95, 1.0, 1.05)):
            C = _vti(v * VP, v * VS, *rs.uniform(0.0, 0.1, 3)) - iso
            for k, (i, j) in enumerate(_PAIRS):
                dC[k, b[m]:b[m + 1]] = C[i, j]
        g = _smooth_noise(shape, gen, 5.0)
        for k, (i, j) in enumerate(_PAIRS):
            if iso[i, j]:
                dC[k] += 0.02 * iso[i, j] * g
    else:                        # random fields: 9 orthorhombic entries, or all 21
        for k, (i, j) in enumerate(_PAIRS):
            if (i, j) in _ORTHO:
                dC[k] = 0.05 * iso[i, j] * _smooth_noise(shape, gen, 5.0)
            elif kind == "full":
                dC[k] = 0.01 * iso[0, 0] * _smooth_noise(shape, gen, 5.0)
        drho.copy_(0.05 * RHO * _smooth_noise(shape, gen, 5.0))
    return dC, drho


def _inputs(case, seed):
    """Everything a case computes with, from the seed alone."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    rs = np.random.RandomState(int(seed) % (2 ** 31))
    n = (case["nx"], case["ny"], case["nz"])
    op = case["op"]
    d = {"n": n, "omega": 2.0 * math.pi * case["freq"] * rs.uniform(0.97, 1.03)}
    d["dC"], d["drho"] = _medium(case, gen, rs)
    # a source off the nodes near the middle, as an event location is
    d["xs"] = [float((0.5 * (v - 1) + rs.uniform(-0.4, 0.4)) * case["dx"]) for v in n]
    M = rs.standard_normal((case["nsrc"], 6))
    d["M"] = M / np.linalg.norm(M, axis=1, keepdims=True)
    if op in ("apply_f64", "apply_f32", "apply_df", "adjoint", "gradient", "frequency"):
        d["u"] = _wavefield(n, gen)
    if op == "apply_f32":
        d["u"] = d["u"].to(torch.complex64)
    if op == "gradient":
        d["lam"] = _wavefield(n, gen)
    if op == "receivers":        # a line of receivers along the surface, and the misfit's residuals
        nr = min(16, n[0])
        d["rec"] = [(int(x), n[1] // 2, 0) for x in np.linspace(0, n[0] - 1, nr)]
        d["freqs"] = [case["freq"] * (1.0 + 0.25 * k) for k in range(case["nsrc"])]
        g = rs.standard_normal((case["nsrc"], nr, 3, 2))
        d["g"] = torch.view_as_complex(torch.from_numpy(g)).cuda()
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    n, op = d["n"], case["op"]
    N = n[0] * n[1] * n[2]
    if op == "receivers":
        s = {"op": op, "g": d["g"]}
        s["model"] = autograd.ReceiverModel(n, case["dx"], LAM, MU, RHO, d["dC"], d["drho"], d["freqs"], d["xs"], d["rec"])
        s["args"] = [d["dC"].requires_grad_(), d["drho"].requires_grad_(),
                     torch.tensor(d["M"][0], dtype=torch.float64, requires_grad=True)]
        return s
    if op in ("apply_f64", "adjoint", "gradient"):
        opts = lsm.lsm_default_opts(precision=lsm.LSM_FP64)
    elif op == "apply_df":
        opts = lsm.lsm_default_opts(precision=lsm.LSM_MIXED, residual=lsm.LSM_RESIDUAL_DFLOAT)
    else:
        opts = lsm.lsm_default_opts(precision=lsm.LSM_MIXED)
    base = d["omega"] if op != "frequency" else 0.8 * d["omega"]
    s = {"op": op, "h": lsm.lsm_create(n, case["dx"], LAM, MU, RHO, d["dC"], d["drho"], base, opts)}
    for k in ("u", "lam"):
        if k in d:
            s[k] = d[k].reshape(-1)
    s.update(xs=d["xs"], M=d["M"].tolist(), omega=d["omega"])
    if op in ("apply_f64", "apply_f32", "apply_df", "adjoint"):
        s["out"] = torch.empty_like(s["u"])
    elif op == "gradient":
        s["gC"] = torch.empty(21 * N, dtype=torch.float64, device="cuda")
        s["grho"] = torch.empty(N, dtype=torch.float64, device="cuda")
    else:
        s["u0"] = [torch.empty(3 * N, dtype=torch.complex128, device="cuda") for _ in range(case["nsrc"])]
        if op == "solve":
            s["x"] = [torch.empty_like(b) for b in s["u0"]]
        else:
            s["out"] = torch.empty_like(s["u0"][0])
    return s


def run(s):
    op, h = s["op"], s.get("h")
    if op == "apply_f64":
        lsm.lsm_apply(h, s["u"], s["out"])
        return s["out"]
    if op == "apply_f32":
        lsm.lsm_apply_c64(h, s["u"], s["out"])
        return s["out"]
    if op == "apply_df":
        lsm.lsm_apply_df(h, s["u"], s["out"])
        return s["out"]
    if op == "adjoint":
        lsm.lsm_adjoint(h, s["u"], s["out"])
        return s["out"]
    if op == "gradient":
        lsm.lsm_gradient(h, s["u"], s["lam"], s["gC"], s["grho"])
        gM = lsm.lsm_source_gradient(h, s["xs"], s["lam"])
        return {"gC": s["gC"], "grho": s["grho"], "gM": np.array(gM)}
    if op == "frequency":
        f = lsm.lsm_create_shared(h, s["omega"])
        lsm.lsm_source_moments(f, s["M"], s["xs"], s["u0"])
        lsm.lsm_apply(f, s["u"], s["out"])
        return {"u0": list(s["u0"]), "Au": s["out"]}
    if op == "solve":
        lsm.lsm_source_moments(h, s["M"], s["xs"], s["u0"])
        for x in s["x"]:
            x.zero_()
        lsm.lsm_solve_batched([h] * len(s["x"]), s["u0"], s["x"])
        return list(s["x"])
    out = s["model"](*s["args"])
    gC, grho, gM = torch.autograd.grad(out, s["args"], s["g"])
    return {"d": out.detach(), "gC": gC, "grho": grho, "gM": gM}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def work(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    N = nx * ny * nz
    NO = (nx + 1) * (ny + 1) * (nz + 1)
    op, k = case["op"], case["nsrc"]
    b = 8 if op == "apply_f32" else 16   # bytes of a complex value
    # one operator application: strain and contraction, divergence and density, three padded FFTs
    # each way with their zero lines left out, the spectral product
    fft = lambda L: 5.0 * L * math.log2(L)  # noqa: E731
    one = 162.0 * N + 54.0 * N + 6.0 * (ny * nz * fft(2 * nx) + 2 * nx * nz * fft(2 * ny) + 4 * nx * ny * fft(2 * nz)) + 66.0 * 8 * N
    medium, spectrum, field = 22 * N * b // 2, 6 * NO * b, 3 * N * b
    if op in ("apply_f64", "apply_f32", "apply_df", "adjoint"):
        return {"bytes": 2 * field + medium + spectrum, "flops": one}
    if op == "gradient":
        return {"bytes": 2 * field + 22 * N * 8 + spectrum, "flops": one}
    if op == "frequency":   # the spectrum is written and read by the application
        table = 6.0 * (4 * ny * nz * fft(2 * nx) + 4 * nx * nz * fft(2 * ny) + 4 * nx * ny * fft(2 * nz)) / 4 + 150.0 * N
        return {"bytes": 2 * spectrum + medium + (2 + k) * field, "flops": one + table + 150.0 * N}
    if op == "solve":       # a few iterations at least; each source's field in, its solution out
        return {"bytes": spectrum + medium + 2 * k * field, "flops": 12.0 * k * one}
    return {"bytes": k * spectrum + 2 * medium, "flops": 2 * 10.0 * k * one}


# ---------------------------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------------------------
def _radial(r, omega):
    """G_ij = f d_ij + g c_i c_j at distance r (c = x / r): f, g and their derivatives."""
    a, b = VP, VS
    ka, kb, c4 = omega / a, omega / b, 1.0 / (4.0 * math.pi * RHO)
    ir = 1.0 / r
    ea, eb = torch.exp(1j * ka * r), torch.exp(1j * kb * r)

    def psi(x, e):   # ((1 - i x) e^{ix} - 1) / x^2
        y = torch.where(x < 0.5, x, torch.full_like(x, 0.5))
        s = torch.zeros_like(e)
        for m in range(17, -1, -1):
            s = s * (1j * y) + (m + 1) / math.factorial(m + 2)
        z = torch.where(x < 0.5, torch.ones_like(x), x)
        return torch.where(x < 0.5, s, ((1 - 1j * z) * e - 1) / (z * z))

    Ea, Eb = ea * ir / a ** 2, eb * ir / b ** 2
    Eap, Ebp = (1j * ka - ir) * Ea, (1j * kb - ir) * Eb
    Q = (psi(kb * r, eb) / b ** 2 - psi(ka * r, ea) / a ** 2) * ir
    Qp = (eb / b ** 2 - ea / a ** 2) * ir * ir - 3.0 * Q * ir
    return c4 * (Eb - Q), c4 * (Ea - Eb + 3 * Q), c4 * (Ebp - Qp), c4 * (Eap - Ebp + 3 * Qp)


def _axis(n, h):
    m = torch.arange(2 * n, device="cuda", dtype=torch.float64)
    return torch.where(m < n, m, m - 2 * n) * h


def _spectrum(case, omega):
    """Spectra of h^3 G (11, 22, 33, 23, 13, 12) on the doubled periodic grid."""
    n, h = (case["nx"], case["ny"], case["nz"]), case["dx"]
    x, y, z = _axis(n[0], h)[None, None, :], _axis(n[1], h)[None, :, None], _axis(n[2], h)[:, None, None]
    r = torch.sqrt(x * x + y * y + z * z)
    r[0, 0, 0] = 1.0
    f, g, _, _ = _radial(r, omega)
    keep = torch.ones_like(r)
    keep[n[2]], keep[:, n[1]], keep[:, :, n[0]] = 0.0, 0.0, 0.0
    # cell average of G over the node's own cell
    C = 3.0 * math.log(2.0 + math.sqrt(3.0)) - 0.5 * math.pi
    c4 = 1.0 / (4.0 * math.pi * RHO)
    self_cell = complex(c4 * (1 / (3 * VP ** 2) + 2 / (3 * VS ** 2)) * C * h * h,
                        c4 * omega * (1 / (3 * VP ** 3) + 2 / (3 * VS ** 3)) * h ** 3)
    out = []
    for i, (p, q) in enumerate(((x, x), (y, y), (z, z), (y, z), (x, z), (x, y))):
        t = g * (p * q / (r * r))
        if i < 3:
            t = t + f
        t = t * (keep * h ** 3)
        t[0, 0, 0] = self_cell if i < 3 else 0.0
        out.append(torch.fft.fftn(t))
        del t
    return out


def _d(f, axis, h):
    """Central difference along an axis of [z, y, x], one-sided at the ends."""
    dim = f.dim() - 1 - axis
    n = f.shape[dim]
    lo, hi = f.narrow(dim, 0, 1), f.narrow(dim, n - 1, 1)
    if n == 2:
        return torch.cat([(hi - lo) / h, (hi - lo) / h], dim)
    mid = (f.narrow(dim, 2, n - 2) - f.narrow(dim, 0, n - 2)) / (2 * h)
    return torch.cat([(f.narrow(dim, 1, 1) - lo) / h, mid, (hi - f.narrow(dim, n - 2, 1)) / h], dim)


_TENSOR = ((0, 5, 4), (5, 1, 3), (4, 3, 2))


def _scattered(case, omega, G, dC, drho, u):
    """u_s = G * (div(dC : eps(u)) + w^2 drho u), u [3, z, y, x]."""
    n, h = (case["nx"], case["ny"], case["nz"]), case["dx"]
    e = [_d(u[0], 0, h), _d(u[1], 1, h), _d(u[2], 2, h), _d(u[1], 2, h) + _d(u[2], 1, h),
         _d(u[0], 2, h) + _d(u[2], 0, h), _d(u[0], 1, h) + _d(u[1], 0, h)]
    at = {p: k for k, p in enumerate(_PAIRS)}
    pad = torch.nn.functional.pad
    sig = [pad(sum(dC[at[min(i, j), max(i, j)]] * e[j] for j in range(6)), (2,) * 6) for i in range(6)]
    core = lambda f, s: f[tuple(slice(1 + v, f.shape[a] - 1 + v) for a, v in enumerate(s))]  # noqa: E731
    q = []
    for j in range(3):
        t = pad(omega ** 2 * drho * u[j], (1,) * 6)
        for k in range(3):
            s = [0, 0, 0]
            s[2 - k] = 1
            S = sig[_TENSOR[j][k]]
            t = t + (core(S, s) - core(S, [-v for v in s])) / (2 * h)
        q.append(torch.fft.fftn(t, s=(2 * n[2], 2 * n[1], 2 * n[0])))
    return torch.stack([torch.fft.ifftn(sum(G[_TENSOR[i][j]] * q[j] for j in range(3)))
                        [1:n[2] + 1, 1:n[1] + 1, 1:n[0] + 1] for i in range(3)])


def _background(case, omega, M, xs):
    """u0_i = -M_jk dG_ij/dx_k of the Voigt moment M."""
    n, h = (case["nx"], case["ny"], case["nz"]), case["dx"]
    ax = [torch.arange(v, device="cuda", dtype=torch.float64) * h - s for v, s in zip(n, xs)]
    X = [ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]]
    r = torch.sqrt(X[0] ** 2 + X[1] ** 2 + X[2] ** 2)
    _, g, fp, gp = _radial(r, omega)
    c = [x / r for x in X]
    m = [[M[_TENSOR[i][j]] for j in range(3)] for i in range(3)]
    Mc = [sum(m[i][j] * c[j] for j in range(3)) for i in range(3)]
    cMc = sum(c[i] * Mc[i] for i in range(3))
    tr = m[0][0] + m[1][1] + m[2][2]
    return torch.stack([-((fp + g / r) * Mc[i] + ((gp - 2 * g / r) * cMc + g / r * tr) * c[i]) for i in range(3)])


def _bicgstab(A, b, tol=2e-14, maxit=400):
    x = torch.zeros_like(b)
    dot = lambda p, q: torch.vdot(p.reshape(-1), q.reshape(-1))  # noqa: E731
    for _ in range(4):           # restarted from the true residual
        r = b - A(x)
        if r.norm() <= tol * b.norm():
            break
        rh, p, rho = r.clone(), r.clone(), dot(r, r)
        stop = max(1e-3 * tol * float(b.norm()), 1e-9 * float(r.norm()))
        for _ in range(maxit):
            v = A(p)
            alpha = rho / dot(rh, v)
            s = r - alpha * v
            t = A(s)
            w = dot(t, s) / dot(t, t)
            x = x + alpha * p + w * s
            r = s - w * t
            if r.norm() <= stop:
                break
            rho, old = dot(rh, r), rho
            p = r + rho / old * (alpha / w) * (p - w * v)
    return x


def exact(case, seed):
    d = _inputs(case, seed)
    op, n = case["op"], d["n"]
    shape = (3, n[2], n[1], n[0])
    w, dC, drho = d["omega"], d["dC"], d["drho"]

    def operator(omega, G):
        return lambda u: u - _scattered(case, omega, G, dC, drho, u)

    def adjoint(omega, G):
        A = operator(omega, G)

        def AH(v):
            with torch.enable_grad():
                u = torch.zeros(shape, dtype=torch.complex128, device="cuda", requires_grad=True)
                return torch.autograd.grad(A(u), u, v)[0]
        return AH

    def gradients(omega, G, u, lam):
        with torch.enable_grad():
            c, r = dC.detach().clone().requires_grad_(), drho.detach().clone().requires_grad_()
            return torch.autograd.grad(_scattered(case, omega, G, c, r, u), (c, r), lam)

    def moments(omega, lam):
        e = np.eye(6)
        return [float((lam.conj() * _background(case, omega, e[j], d["xs"])).real.sum()) for j in range(6)]

    with torch.no_grad():
        if op == "receivers":
            out, gC, grho, gM = [], 0.0, 0.0, np.zeros(6)
            rec = torch.tensor([(z * n[1] + y) * n[0] + x for x, y, z in d["rec"]], device="cuda")
            for k, f in enumerate(d["freqs"]):
                om = 2.0 * math.pi * f
                G = _spectrum(case, om)
                u = _bicgstab(operator(om, G), _background(case, om, d["M"][0], d["xs"]))
                out.append(u.reshape(3, -1)[:, rec].transpose(0, 1))
                rhs = torch.zeros((3, u[0].numel()), dtype=torch.complex128, device="cuda")
                rhs[:, rec] = d["g"][k].transpose(0, 1)
                lam = _bicgstab(adjoint(om, G), rhs.reshape(shape))
                a, b = gradients(om, G, u, lam)
                gC, grho, gM = gC + a, grho + b, gM + np.array(moments(om, lam))
            return {"d": torch.stack(out), "gC": gC, "grho": grho, "gM": torch.from_numpy(gM)}
        G = _spectrum(case, w)
        if op in ("apply_f64", "apply_f32", "apply_df"):
            return operator(w, G)(d["u"].to(torch.complex128)).reshape(-1)
        if op == "adjoint":
            return adjoint(w, G)(d["u"]).reshape(-1)
        if op == "gradient":
            gC, grho = gradients(w, G, d["u"], d["lam"])
            return {"gC": gC.reshape(-1), "grho": grho.reshape(-1), "gM": np.array(moments(w, d["lam"]))}
        u0 = [_background(case, w, m, d["xs"]) for m in d["M"]]
        if op == "frequency":
            return {"u0": [b.reshape(-1) for b in u0], "Au": operator(w, G)(d["u"]).reshape(-1)}
        return [_bicgstab(operator(w, G), b).reshape(-1) for b in u0]
