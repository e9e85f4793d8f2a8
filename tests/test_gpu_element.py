"""GPU parity: FP32 products evaluated element by element against the oracle.

Sizes cover one partly filled block of 32 cubes (n = 2, 3), whole blocks (4),
blocks that straddle x-lines and a ragged last block (5, 9, 13). The bound
counts roundings: every result is a sum of at most 24 element terms of about
30 FP32 operations each whose operands are of the size of |M||x|, so 32 units
of rounding of that vector bound the error in norm.
"""

import numpy as np
import pytest

import workload as wl
from oracle.assemble import StokesSystem
from oracle.mesh import KuhnMesh

from gpu_helpers import aos, cuda, gpu_module, host, soa

pytestmark = pytest.mark.gpu

BOUND = 32 * 2.0 ** -24


@pytest.mark.parametrize("n,mu,dt", [(2, 0.3, 0.05), (3, 1e-4, 1e-4), (4, 1.0, 1e-2), (5, 1e-2, 1e-3),
                                     (9, 1.0, 1e-2), (13, 1e-3, 1e-3)])
def test_fp32_strain_product(n, mu, dt):
    sk = gpu_module()
    V = wl.kuhn_vertices(n, 0.16, 7)
    S = sk.Stokes(n, V, mu, dt, 0.0, sk.stokes_default_options(precision=1))
    orc = StokesSystem(KuhnMesh(n, V), mu, dt)
    x = np.random.default_rng(n).standard_normal(orc.A.shape[1]).astype(np.float32).astype(np.float64)
    y = aos(host(S.apply("A_F32", cuda(soa(x)), x.size)))
    assert np.linalg.norm(y - orc.A @ x) <= BOUND * np.linalg.norm(abs(orc.A) @ abs(x))
    again = aos(host(S.apply("A_F32", cuda(soa(x)), x.size)))
    assert np.array_equal(y, again)
    S.close()
