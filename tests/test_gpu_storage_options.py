"""GPU: mixed-precision solves under the options that decide which matrices
products read from CSR, from stencil storage or not at all.

Setup makes FP32 CSR copies only where a product reads them; every option that
does read them is run here on an odd and a nested hierarchy (34: the restriction
from CSR, 17 below it without), one and four right-hand sides, against the
default storage. Solutions to 1e-10 of one system agree to 1e-8.
"""

import numpy as np
import pytest

import workload as wl

from gpu_helpers import cuda, gpu_module, host, rel_err

pytestmark = pytest.mark.gpu


def _solve(n, f, **opts):
    sk = gpu_module()
    S = sk.Stokes(n, wl.kuhn_vertices(n, 0.16, 2), 1e-2, 1e-3, 0.0,
                  sk.stokes_default_options(precision=1, vcycles=1, max_refine=12, **opts))
    u, _, _ = S.solve(cuda(f[0]), None, 1e-10)
    U, _, _ = S.solve_multi(cuda(f), None, 1e-10)
    S.close()
    return host(u), host(U)


@pytest.mark.parametrize("n", [9, 34])
@pytest.mark.parametrize("method", [0, 1])
def test_storage_options(n, method):
    f = np.stack([wl.random_force(n, 70 + k).reshape(-1, 3) for k in range(4)])
    u0, U0 = _solve(n, f, method=method)
    for opts in (dict(coarse_kernel=1), dict(stencil_min_rows=3000), dict(format=1), dict(format=2), dict(format=3),
                 dict(schur_prec=2), dict(vel_prec=2), dict(spmv_group=4), dict(vcycle_split=2), dict(vcycle_split=0)):
        u, U = _solve(n, f, method=method, **opts)
        assert rel_err(u, u0) <= 1e-8 and rel_err(U, U0) <= 1e-8, opts
