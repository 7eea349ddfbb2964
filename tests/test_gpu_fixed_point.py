"""The FP64 operator's fixed-point transforms (csrc/fx.cuh) where their scaling can go wrong.

* Every line is scaled by a power of two, so scaling a field by one scales the result exactly.
* A line's unit follows its largest value: rows, columns and components of very different sizes
  still meet the FP64 parity tolerance (1e-12: FP64 rounding grows like u log2(P), about 2e-15).
* A zero field stays exactly zero; an infinity or a NaN anywhere makes every output NaN, as the
  transforms of any arithmetic do (each output sums over all inputs).
"""
import numpy as np
import pytest
import torch

import synthetic as sy
from oracle import operator as op
from paper_2301_12836_gb300 import lsm

from gpu_helpers import dev, field, handle, host, rel

pytestmark = pytest.mark.gpu

W = 2 * np.pi * 9.0
# every compile-time line length (16 .. 512) on every axis, beside generic ones
# (512, that is sides of 256, in test_gpu_fixed_point_long.py)
GRIDS = [(8, 16, 32), (32, 8, 16), (16, 32, 8), (64, 9, 8), (12, 64, 10), (8, 10, 64), (128, 8, 9), (9, 128, 8), (8, 9, 128)]


def _apply(h, u, adjoint=False):
    out = torch.empty(3 * h.N, dtype=torch.complex128, device="cuda")
    (lsm.lsm_adjoint if adjoint else lsm.lsm_apply)(h, dev(u).reshape(-1), out)
    return host(out).reshape(u.shape)


@pytest.mark.parametrize("n", GRIDS)
def test_scaling_by_powers_of_two_is_exact(n):
    med = sy.random_medium(n, h=8.0, seed=sum(n), frac=0.2)
    h = handle(med, W)
    u = field(med.shape, 7)
    want, want_h = _apply(h, u), _apply(h, u, True)
    for k in (-600, -40, 300):
        s = 2.0 ** k
        assert np.array_equal(_apply(h, u * s), want * s)
        assert np.array_equal(_apply(h, u * s, True), want_h * s)


@pytest.mark.parametrize("n", GRIDS)
def test_uneven_fields(n):
    """A field that falls by eight decades along every axis and between components, and one with a
    single entry."""
    med = sy.random_medium(n, h=8.0, seed=sum(n) + 1, frac=0.2)
    h = handle(med, W)
    F = op.FFTOperator(med, W)
    z, y, x = np.meshgrid(*[np.linspace(0, 1, s) for s in med.shape], indexing="ij")
    u = field(med.shape, 8) * 10.0 ** (-8 * (x + y + z)) * np.array([1.0, 1e-4, 1e-8])[:, None, None, None]
    one = np.zeros_like(u)
    one[1, n[2] // 2, n[1] // 2, n[0] // 2] = 1.0 - 2.0j
    for v in (u, one):
        assert rel(_apply(h, v), F.apply(v)) < 1e-12
        assert rel(_apply(h, v, True), F.adjoint(v)) < 1e-12


@pytest.mark.parametrize("n", [(8, 16, 32), (64, 9, 8), (8, 9, 128)])
def test_zero_infinite_and_nan_fields(n):
    med = sy.random_medium(n, h=8.0, seed=sum(n) + 2, frac=0.2)
    h = handle(med, W)
    u = field(med.shape, 9)
    assert not np.any(_apply(h, np.zeros_like(u)))
    tiny = _apply(h, u * 2.0 ** -1060)
    assert np.all(np.isfinite(tiny.view(np.float64)))
    for bad in (np.nan, np.inf):
        v = u.copy()
        v[2, n[2] // 2, n[1] // 3, n[0] // 3] = bad
        assert np.all(np.isnan(_apply(h, v)))


# generic lengths: every radix first and last, one-stage plans, the longest line, tile remainders
GENERIC = [(2, 3, 4), (5, 6, 10), (9, 15, 25), (27, 12, 45), (50, 81, 6), (6, 125, 9), (10, 9, 125), (250, 3, 4), (4, 250, 3),
           (3, 4, 250), (96, 5, 12), (5, 96, 4), (12, 5, 96)]


@pytest.mark.parametrize("n", GENERIC)
def test_generic_lengths(n):
    """Forward and adjoint operators against the oracle, and the exact scaling, on lines of the
    runtime engine."""
    med = sy.random_medium(n, h=8.0, seed=sum(n) + 3, frac=0.2)
    h = handle(med, W)
    F = op.FFTOperator(med, W)
    u = field(med.shape, 10)
    got, got_h = _apply(h, u), _apply(h, u, True)
    assert rel(got, F.apply(u)) < 1e-12
    assert rel(got_h, F.adjoint(u)) < 1e-12
    assert np.array_equal(_apply(h, u * 2.0 ** -500), got * 2.0 ** -500)
    assert not np.any(_apply(h, np.zeros_like(u)))


@pytest.mark.parametrize("v", [1, 2])
def test_generic_engine_on_two_step_lengths(v):
    """The schedule's generic variants of 16 .. 256: within rounding of the default kernels."""
    for n in ((8, 16, 32), (64, 8, 8), (8, 9, 128)):
        med = sy.random_medium(n, h=8.0, seed=sum(n) + 4, frac=0.2)
        h = handle(med, W)
        u = field(med.shape, 11)
        want = _apply(h, u)
        lsm.lsm_set_schedule(h, lsm.LSM_FP64, [0, v, v, v, v, v])
        assert rel(_apply(h, u), want) < 2e-14
