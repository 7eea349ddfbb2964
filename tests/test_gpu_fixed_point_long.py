"""The FP64 operator's fixed-point transforms on 512-point lines (sides of 256), along each axis, and its
accuracy on a side of every two-step length and on long lines of the runtime engine.

Accuracy, per displacement component, forward and adjoint: the distance from the longdouble value is
at most twice that of a NumPy evaluation of the same formulas in FP64 (the two differ in the order of
their roundings; a scaling that lost a bit on every line would show as a factor of two by itself).
"""
import numpy as np
import pytest
import torch

import extended as ext
import synthetic as sy
from paper_2301_12836_gb300 import lsm

from gpu_helpers import dev, field, handle, host

pytestmark = pytest.mark.gpu

LONG = [(256, 5, 6), (5, 256, 6), (6, 5, 256)]
GENERIC = [(81, 5, 6), (5, 125, 6), (6, 5, 144), (180, 5, 4), (5, 225, 4), (4, 5, 250), (243, 4, 5), (5, 4, 240)]
SIDES = [(8, 16, 32), (64, 9, 8), (8, 128, 9)] + LONG


def _apply(h, u, adjoint=False):
    out = torch.empty(3 * h.N, dtype=torch.complex128, device="cuda")
    (lsm.lsm_adjoint if adjoint else lsm.lsm_apply)(h, dev(u).reshape(-1), out)
    return host(out).reshape(u.shape)


def _setup(n, seed):
    med = sy.random_medium(n, h=8.0, seed=sum(n) + seed, frac=0.2)
    med.dC, med.drho = 30 * med.dC, 30 * med.drho   # the scattered part makes up most of A u
    w = 2 * np.pi * np.sqrt(med.mu0 / med.rho0) / (8.0 * max(n))   # one shear wavelength per longest side
    return med, w


@pytest.mark.parametrize("n", SIDES + GENERIC)
def test_components_against_longdouble(n):
    med, w = _setup(n, 51)
    h = handle(med, w)
    assert np.finfo(np.longdouble).nmant >= 63
    G = {R: ext.spectrum(med, w, R) for R in (np.longdouble, np.float64)}
    z, y, x = np.meshgrid(*[np.linspace(0, 1, s) for s in med.shape], indexing="ij")
    white = field(med.shape, 21)
    decaying = white * 10.0 ** (-8 * (x + y + z)) * np.array([1.0, 1e-4, 1e-8])[:, None, None, None]
    plane = np.exp(2j * np.pi * (x + 0.5 * y + 0.25 * z)) * np.array([1.0, -2.0, 0.5])[:, None, None, None]
    for u in (white, decaying, plane):
        for f in (ext.apply, ext.adjoint):
            exact, fp64 = (f(med, w, G[R], u, R) for R in (np.longdouble, np.float64))
            got = _apply(h, u, f is ext.adjoint)
            for c in range(3):
                size = np.linalg.norm(exact[c].astype(np.complex128))
                err = [np.linalg.norm((a[c] - exact[c]).astype(np.complex128)) / size for a in (got, fp64)]
                assert err[0] <= 2 * err[1], (c, f.__name__)


@pytest.mark.parametrize("n", LONG)
def test_long_lines_scale_exactly(n):
    med, w = _setup(n, 52)
    h = handle(med, w)
    u = field(med.shape, 22)
    want, want_h = _apply(h, u), _apply(h, u, True)
    for k in (-600, -40, 300):
        s = 2.0 ** k
        assert np.array_equal(_apply(h, u * s), want * s)
        assert np.array_equal(_apply(h, u * s, True), want_h * s)


@pytest.mark.parametrize("n", LONG)
def test_long_lines_zero_infinite_and_nan(n):
    med, w = _setup(n, 53)
    h = handle(med, w)
    u = field(med.shape, 23)
    assert not np.any(_apply(h, np.zeros_like(u)))
    for bad in (np.nan, np.inf):
        v = u.copy()
        v[2, n[2] // 2, n[1] // 3, n[0] // 3] = bad
        assert np.all(np.isnan(_apply(h, v)))


def test_subnormal_results():
    """A field of 2^-1035: the displacements, and the transforms' intermediates that stand for them, lie
    below the normal range, where a value keeps 2^-1074.  Relative to u that is 2^-39; the strain's
    1 / 2h, the spectrum's 1 / P and the sums over a line lose at most 12 bits more.  (The adjoint's
    first intermediate is about 2^-30 u, the kernel before the contrast: there FP64 itself keeps 9 bits.)"""
    n = (8, 16, 32)
    med, w = _setup(n, 54)
    h = handle(med, w)
    u = field(med.shape, 24)
    s = 2.0 ** -1035
    scattered = u - _apply(h, u)
    got = (u * s - _apply(h, u * s)) * 2.0 ** 600 * 2.0 ** 435   # 1 / s is out of range
    assert np.linalg.norm(got - scattered) < 2.0 ** -27 * np.linalg.norm(scattered)
