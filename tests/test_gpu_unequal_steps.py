"""FP32 passes of the line lengths L = A * B with B = 2 A (32, 128, 512; node counts 16, 64, 256): the
register-resident z pass and the warp-per-line x passes, along each axis and with row and column
counts that leave their blocks ragged, against the FP64 apply of the same field.

Tolerance: rounding of six transforms of at most nine radix-2 layers and of the node kernels, each
2^-24 of the values' norm at most when all errors add up: (6 * 9 + 10) 2^-24 = 3.8e-6.
"""
import numpy as np
import pytest
import torch

import synthetic as sy

from gpu_helpers import dev, field, handle, host, rel
from paper_2301_12836_gb300 import lsm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(16, 5, 3), (3, 5, 16), (64, 3, 5), (5, 3, 64), (256, 5, 3), (2, 3, 256), (16, 64, 16), (64, 9, 64)])
def test_fp32_apply_against_fp64(n):
    med = sy.random_medium(n, h=8.0, seed=sum(n) + 31, frac=0.2)
    h = handle(med, 2 * np.pi * 10.0, precision=lsm.LSM_MIXED)
    u = field(med.shape, 15).astype(np.complex64)
    A32 = torch.empty(3 * h.N, dtype=torch.complex64, device="cuda")
    A64 = torch.empty(3 * h.N, dtype=torch.complex128, device="cuda")
    lsm.lsm_apply_c64(h, dev(u, torch.complex64).reshape(-1), A32)
    lsm.lsm_apply(h, dev(u.astype(np.complex128)).reshape(-1), A64)
    a32, a64 = host(A32).reshape(u.shape).astype(np.complex128), host(A64).reshape(u.shape)
    assert rel(a32, a64) < 64 * 2.0 ** -24
    assert rel(u.astype(np.complex128), a64) > 1e-3
