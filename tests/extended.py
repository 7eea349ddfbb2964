"""The operator and its adjoint in a chosen real type (NumPy longdouble: the exact value the FP64
operator approximates; float64: the yardstick of what FP64 rounding leaves).

The kernel table's near-field terms come from their power series, so the table loses no digits at
distances far below a wavelength (the closed forms of ``oracle.green`` cancel there).
"""
import math

import numpy as np
import scipy.fft as sf

T2V = ((0, 5, 4), (5, 1, 3), (4, 3, 2))
PLANE = {p: k for k, p in enumerate((i, j) for i in range(6) for j in range(i, 6))}


def complex_type(R):
    return np.result_type(R, np.complex64)


def _psi(x, e):
    """((1 - i x) e^{ix} - 1) / x^2, by its series below 1/2."""
    R = x.dtype.type
    y = np.where(x < 0.5, x, R(0.5))
    s = np.zeros(x.shape, complex_type(R))
    for m in range(23, -1, -1):
        s = s * (1j * y) + R(m + 1) / R(math.factorial(m + 2))
    z = np.where(x < 0.5, R(1), x)
    return np.where(x < 0.5, s, ((1 - 1j * z) * e - 1) / (z * z))


def spectrum(med, w, R):
    """Spectrum of the kernel table, six planes [2nz, 2ny, 2nx] (order 11, 22, 33, 23, 13, 12)."""
    pi, h, w = R("3.14159265358979323846264338327950288") if R is np.longdouble else R(np.pi), R(med.h), R(w)
    rho = R(med.rho0)
    a, b = np.sqrt((R(med.lam0) + 2 * R(med.mu0)) / rho), np.sqrt(R(med.mu0) / rho)
    nx, ny, nz = med.n

    def axis(m):
        v = np.arange(2 * m).astype(R)
        return np.where(v < m, v, v - 2 * m) * h
    x, y, z = axis(nx)[None, None, :], axis(ny)[None, :, None], axis(nz)[:, None, None]
    r = np.sqrt(x * x + y * y + z * z)
    r[0, 0, 0] = 1
    c4, ir = 1 / (4 * pi * rho), 1 / r
    ea, eb = (np.cos(k * r) + 1j * np.sin(k * r) for k in (w / a, w / b))
    Ea, Eb = ea * ir / (a * a), eb * ir / (b * b)
    Q = (_psi(w / b * r, eb) / (b * b) - _psi(w / a * r, ea) / (a * a)) * ir
    f, g = c4 * (Eb - Q), c4 * (Ea - Eb + 3 * Q)
    keep = np.ones(r.shape, R) * h ** 3
    keep[nz], keep[:, ny], keep[:, :, nx] = 0, 0, 0
    cube = 3 * np.log(2 + np.sqrt(R(3))) - pi / 2
    own = c4 * (1 / (3 * a * a) + 2 / (3 * b * b)) * cube * h * h + 1j * c4 * w * (1 / (3 * a ** 3) + 2 / (3 * b ** 3)) * h ** 3
    out = []
    for i, (p, q) in enumerate(((x, x), (y, y), (z, z), (y, z), (x, z), (x, y))):
        t = (g * (p * q / (r * r)) + (f if i < 3 else 0)) * keep
        t[0, 0, 0] = own if i < 3 else 0
        out.append(sf.fftn(t))
    return out


def _d(f, a, h):
    """Central difference along coordinate a (0 = x), one-sided at the ends."""
    f = np.moveaxis(f, 2 - a, -1)
    o = np.empty_like(f)
    o[..., 1:-1] = (f[..., 2:] - f[..., :-2]) / (2 * h)
    o[..., 0], o[..., -1] = (f[..., 1] - f[..., 0]) / h, (f[..., -1] - f[..., -2]) / h
    return np.moveaxis(o, -1, 2 - a)


def _dt(f, a, h):
    """Transpose of ``_d``."""
    f = np.moveaxis(f, 2 - a, -1)
    o = np.zeros_like(f)
    o[..., 2:] += f[..., 1:-1] / (2 * h)
    o[..., :-2] -= f[..., 1:-1] / (2 * h)
    o[..., 1] += f[..., 0] / h
    o[..., 0] -= f[..., 0] / h
    o[..., -1] += f[..., -1] / h
    o[..., -2] -= f[..., -1] / h
    return np.moveaxis(o, -1, 2 - a)


def _contract(dC, e):
    return [sum(dC[PLANE[min(i, j), max(i, j)]] * e[j] for j in range(6)) for i in range(6)]


def _shifted(f, a, s):
    """f less its outermost nodes, read s nodes along coordinate a."""
    sl = [slice(1, -1)] * 3
    sl[2 - a] = slice(1 + s, f.shape[2 - a] - 1 + s)
    return f[tuple(sl)]


def apply(med, w, G, u, R):
    nx, ny, nz = med.n
    h, w, u = R(med.h), R(w), u.astype(complex_type(R))
    dC, drho = med.dC.astype(R), med.drho.astype(R)
    e = [_d(u[0], 0, h), _d(u[1], 1, h), _d(u[2], 2, h), _d(u[1], 2, h) + _d(u[2], 1, h),
         _d(u[0], 2, h) + _d(u[2], 0, h), _d(u[0], 1, h) + _d(u[1], 0, h)]
    sig = [np.pad(s, 2) for s in _contract(dC, e)]
    Q = []
    for j in range(3):
        q = np.pad(w ** 2 * drho * u[j], 1)
        for k in range(3):
            q = q + (_shifted(sig[T2V[j][k]], k, 1) - _shifted(sig[T2V[j][k]], k, -1)) / (2 * h)
        Q.append(sf.fftn(q, s=(2 * nz, 2 * ny, 2 * nx)))
    return u - np.stack([sf.ifftn(sum(G[T2V[i][j]] * Q[j] for j in range(3)))[1:nz + 1, 1:ny + 1, 1:nx + 1] for i in range(3)])


def adjoint(med, w, G, v, R):
    nx, ny, nz = med.n
    h, w, v = R(med.h), R(w), v.astype(complex_type(R))
    dC, drho = med.dC.astype(R), med.drho.astype(R)
    V = []
    for c in range(3):
        p = np.zeros((2 * nz, 2 * ny, 2 * nx), v.dtype)
        p[1:nz + 1, 1:ny + 1, 1:nx + 1] = v[c]
        V.append(sf.fftn(p))
    z = [sf.ifftn(sum(np.conj(G[T2V[i][j]]) * V[j] for j in range(3)))[:nz + 2, :ny + 2, :nx + 2] for i in range(3)]
    tau = [0] * 6
    for j in range(3):
        for k in range(3):
            tau[T2V[j][k]] = tau[T2V[j][k]] + (_shifted(z[j], k, -1) - _shifted(z[j], k, 1)) / (2 * h)
    c = _contract(dC, tau)
    return np.stack([v[i] - sum(_dt(c[T2V[i][a]], a, h) for a in range(3)) - w ** 2 * drho * z[i][1:-1, 1:-1, 1:-1] for i in range(3)])
