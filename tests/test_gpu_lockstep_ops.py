"""GPU: the building blocks of the FP32 lockstep solves (four systems at once)
against the same operators on one system, the oracle and FP64.

The element product gives every system the bits of the product on its own, with
several systems per launch (up to 41 cubes) and one per launch (from 42 on). B
and B^T with their addend and scaling are held to 32 units of rounding of the
sums of magnitudes, as the products on one system. A V-cycle in FP32 (some 30
sweeps of sums of up to 65 terms, 8 units each) is held to 256 units of rounding
of its result, C, which inverts an operator of condition about 10^3, to 4096.
The V-cycle sizes lie on both sides of the lines at which a row's entries go
over 8, 4 and 2 warps (2^15, 2^16, 2^18, 2^19 rows) and below them on the
coarser levels, nested and odd.
"""

import numpy as np
import pytest

import workload as wl
from oracle.assemble import StokesSystem
from oracle.mesh import KuhnMesh

from gpu_helpers import aos, cuda, gpu_module, host, soa

pytestmark = pytest.mark.gpu

UNIT = 2.0 ** -24


def _setup(n, **opts):
    sk = gpu_module()
    V = wl.kuhn_vertices(n, 0.16, 3)
    return V, sk.Stokes(n, V, 1e-2, 1e-3, 0.0, sk.stokes_default_options(precision=1, **opts))


def _f32(rng, *shape):
    return rng.standard_normal(shape).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("n", [2, 9, 13, 41, 42])
def test_strain_product(n):
    _, S = _setup(n)
    nv = 3 * S.sizes["n_inner"]
    x, b = _f32(np.random.default_rng(n), 2, 4, nv)
    y = host(S.apply("A_F32_X4", cuda(np.stack([x, b]).ravel()), 8 * nv + 4))
    Ax, res, dots = y[:4 * nv].reshape(4, nv), y[4 * nv:8 * nv].reshape(4, nv), y[8 * nv:]
    for k in range(4):
        one = host(S.apply("A_F32", cuda(x[k]), nv))
        assert np.array_equal(Ax[k], one)
        assert np.array_equal(res[k], (b[k].astype(np.float32) - one.astype(np.float32)).astype(np.float64))
        assert abs(dots[k] - x[k] @ one) <= 2.0 ** -40 * (abs(x[k]) @ abs(one))
    S.close()


@pytest.mark.parametrize("n", [2, 3, 9, 14])
def test_divergence(n):
    V, S = _setup(n)
    orc = StokesSystem(KuhnMesh(n, V), 1e-2, 1e-3)
    nv, npr = orc.A.shape[0], orc.B.shape[0]
    rng = np.random.default_rng(n)
    u, bu, q, bq = _f32(rng, 4, nv), _f32(rng, 4, nv), _f32(rng, 4, npr), _f32(rng, 4, npr)
    r = host(S.apply("B_F32_X4", cuda(np.concatenate([np.stack([soa(v) for v in u]).ravel(), bq.ravel()])), 4 * npr))
    w = host(S.apply("BT_F32_X4", cuda(np.concatenate([q.ravel(), np.stack([soa(v) for v in bu]).ravel()])), 4 * nv))
    for k in range(4):
        want = bq[k] - orc.B @ u[k]
        size = abs(bq[k]) + abs(orc.B) @ abs(u[k])
        assert np.linalg.norm(r.reshape(4, -1)[k] - want) <= 32 * UNIT * np.linalg.norm(size)
        want = bu[k] - (orc.B.T @ q[k]) / orc.Lam
        size = abs(bu[k]) + (abs(orc.B.T) @ abs(q[k])) / orc.Lam
        assert np.linalg.norm(aos(w.reshape(4, -1)[k]) - want) <= 32 * UNIT * np.linalg.norm(size)
    S.close()


def _four_and_one(S, op, x, units):
    length = x.shape[1]
    four = host(S.apply(op + "_F32_X4", cuda(x.ravel()), 4 * length)).reshape(4, length)
    for k in range(4):
        one = host(S.apply(op + "_F32", cuda(x[k]), length))
        want = host(S.apply(op, cuda(x[k]), length))
        size = np.linalg.norm(want)
        assert np.linalg.norm(one - want) <= units * UNIT * size
        assert np.linalg.norm(four[k] - want) <= units * UNIT * size


@pytest.mark.parametrize("n,split", [(4, 1), (7, 1), (8, 0), (16, 1), (17, 0), (20, 1), (21, 1), (32, 1), (33, 1),
                                     (40, 1), (41, 1)])
def test_velocity_cycle(n, split):
    _, S = _setup(n, vcycles=1, vcycle_split=split)
    _four_and_one(S, "VCYCLE_VEL", _f32(np.random.default_rng(n), 4, 3 * S.sizes["n_inner"]), 256)
    S.close()


@pytest.mark.parametrize("n", [5, 12, 17])
def test_schur_preconditioner(n):
    _, S = _setup(n)
    _four_and_one(S, "SCHUR_PREC", _f32(np.random.default_rng(n), 4, S.sizes["n_p1"]), 4096)
    S.close()
