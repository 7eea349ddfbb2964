"""Solves whose length is chaotic, checked by what rounding cannot decide.

BiCGSTAB amplifies a perturbation of 1e-15 in every operator application (layers64, 15 Hz, oracle) to
7e-13 in the eighth iterate, 2e-9 in the sixteenth and to order one in the count: solves of the same
system scaled by factors in [1, 2) took 166 to 458 iterations (oracle: 216).  So a count is not
compared with another count; the eighth iterate is compared with the oracle's, within 150 times the
amplified perturbation, and the median count over nine scaled systems lies within 30% of the oracle's.
"""
import os

import numpy as np
import pytest
import torch

import synthetic as sy
from oracle import operator as op, solver as osv, source as osrc
from paper_2301_12836_gb300 import lsm

from gpu_helpers import dev, handle, host, rel

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

W = 2 * np.pi * 15.0
ORACLE_COUNT = 216


@pytest.fixture(scope="module")
def layers64():
    wl = sy.get_workload("layers64")
    M, xs = wl.sources()
    return wl.medium(), M[0], xs[0]


def test_layers64_eighth_iterate(layers64):
    med, M, xs = layers64
    F = op.FFTOperator(med, W, workers=os.cpu_count() or 1)
    u0, _ = osrc.background_field(med.n, med.h, M, xs, W, med.lam0, med.mu0, med.rho0)
    want, it, rr, status, _ = osv.bicgstab(F.apply, u0, tol=1e-12, maxit=8)
    assert status == osv.NOCONV and it == 8
    h = handle(med, W, tol=1e-12, maxit=8)
    x = torch.zeros(3 * h.N, dtype=torch.complex128, device="cuda")
    code, got_it, got_rr = lsm.lsm_solve(h, dev(u0).reshape(-1), x, check=False)
    assert code == lsm.LSM_ERR_NOCONV and got_it == 8
    assert rel(host(x).reshape(u0.shape), want) < 1e-10
    assert abs(got_rr - rr) < 1e-10


def test_layers64_median_count(layers64):
    med, M, xs = layers64
    h = handle(med, W, tol=1e-12, maxit=2000)
    b = torch.empty(3 * h.N, dtype=torch.complex128, device="cuda")
    lsm.lsm_source(h, M, xs, b)
    counts = []
    for s in np.random.default_rng(2).uniform(1.0, 2.0, 9):
        x = torch.zeros_like(b)
        code, it, rr = lsm.lsm_solve(h, b * float(s), x)
        assert code == lsm.LSM_OK and rr <= 1e-12
        counts.append(it)
    assert abs(np.median(counts) - ORACLE_COUNT) <= 0.3 * ORACLE_COUNT, counts
