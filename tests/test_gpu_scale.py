"""GPU: solves of forces far from unit size in mixed precision.

A force times a power of two has the solution times the same power of two: the
load, the FP64 residuals and every coefficient of the Krylov methods scale
exactly, and the FP32 corrections run on a residual brought to unit norm, so
the two solutions are equal bit for bit, however large or small the force while the
FP32 pairs of the refinement residual stay in range (2^73, about 1e22: sums of
squares of its load do not).
"""

import numpy as np
import pytest

import workload as wl

from gpu_helpers import cuda, gpu_module, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", [0, 1])
@pytest.mark.parametrize("exponent", [73, 110, -40])
def test_scaled_force(method, exponent):
    sk = gpu_module()
    n = 8
    S = sk.Stokes(n, wl.kuhn_vertices(n, 0.16, 4), 1e-2, 1e-3, 0.0,
                  sk.stokes_default_options(precision=1, vcycles=1, method=method, max_refine=12))
    f = wl.random_force(n, 5).reshape(-1, 3)
    u, p, _ = S.solve(cuda(f), None, 1e-10)
    us, ps, info = S.solve(cuda(np.ldexp(f, exponent)), None, 1e-10)
    assert info.status == 0 and info.rel_residual <= 1e-10
    assert np.array_equal(host(us), np.ldexp(host(u), exponent))
    assert np.array_equal(host(ps), np.ldexp(host(p), exponent))
    S.close()


@pytest.mark.parametrize("method", [0, 1])
def test_scaled_forces_in_one_group(method):
    """Each system of a lockstep group has its own scale."""
    sk = gpu_module()
    n = 8
    S = sk.Stokes(n, wl.kuhn_vertices(n, 0.16, 4), 1e-2, 1e-3, 0.0,
                  sk.stokes_default_options(precision=1, vcycles=1, method=method, max_refine=12))
    F = np.stack([wl.random_force(n, 6 + k).reshape(-1, 3) for k in range(4)])
    e = np.array([73, 0, -40, 110]).reshape(4, 1, 1)
    U, P, _ = S.solve_multi(cuda(F), None, 1e-10)
    Us, Ps, infos = S.solve_multi(cuda(np.ldexp(F, e)), None, 1e-10)
    assert all(i.status == 0 and i.rel_residual <= 1e-10 for i in infos)
    assert np.array_equal(host(Us), np.ldexp(host(U), e))
    assert np.array_equal(host(Ps), np.ldexp(host(P), e[:, 0]))
    S.close()
