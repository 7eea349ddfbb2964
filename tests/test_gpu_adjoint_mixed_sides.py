"""Mixed-precision adjoint solves on sides whose x lines have two-step kernels (2 nx = 16 .. 512).  The FP32
adjoint's x passes have an input offset and an inverse direction, which the FP32 two-step row kernels do
not: the launcher must send them to the runtime engine, whatever the caller asks for.

The bar is that of the mixed forward solves against FP64 ones: 1e-6 at a tolerance of 1e-8.
"""
import numpy as np
import pytest
import torch

import synthetic as sy
from paper_2301_12836_gb300 import lsm

from gpu_helpers import dev, field, handle, host, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(8, 6, 5), (16, 5, 6), (32, 6, 5), (64, 5, 6), (128, 5, 6), (256, 5, 6)])
def test_mixed_adjoint_solve_against_fp64(n):
    med = sy.random_medium(n, h=8.0, seed=sum(n) + 61, frac=0.2)
    b = dev(field(med.shape, 31)).reshape(-1)
    xs = []
    for precision, tol in ((lsm.LSM_FP64, 1e-11), (lsm.LSM_MIXED, 1e-8)):
        h = handle(med, 2 * np.pi * 9.0, precision=precision, tol=tol, maxit=2000)
        x = torch.zeros_like(b)
        lsm.lsm_solve_adjoint(h, b, x)
        xs.append(host(x))
    assert rel(xs[1], xs[0]) < 1e-6
