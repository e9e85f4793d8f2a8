"""GPU: launch counts that the library reports for the P2 transfers.

One transfer is one launch, on both sides of the line (32 cubes, nested) up to
which the FP32 restriction runs without its matrix.
"""

import numpy as np
import pytest

import workload as wl

from gpu_helpers import cuda, gpu_module

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [7, 32, 34])
def test_transfer_counts(n):
    sk = gpu_module()
    S = sk.Stokes(n, wl.kuhn_vertices(n, 0.1, 1), 1e-2, 1e-3, 0.0,
                  sk.stokes_default_options(precision=1, profile=1))
    nf, nc = 3 * (2 * n - 1) ** 3, 3 * (2 * ((n + 1) // 2) - 1) ** 3
    for op, nx, ny in (("RESTRICT_P2_F32", nf, nc), ("PROLONG_P2_F32", nc, nf)):
        sk.stokes_kernel_stats_reset(S.ctx)
        S.apply(op, cuda(np.ones(nx)), ny)
        launches, _, nbytes = S.kernel_stats("TRANSFER")
        assert launches == 1
        assert nbytes >= 4 * (nx + ny)
    S.close()
