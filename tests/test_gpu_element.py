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

from gpu_helpers import aos, cuda, gpu_module, host, soa, to_scipy

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


@pytest.mark.parametrize("n", [2, 3, 5, 9, 14])
def test_divergence_stencil(n):
    """B and B^T from the shared stencil storage (n = 2, 3: offsets that alias
    in the linear index; 14: several blocks per parity class), both precisions.
    A row sums at most 65 x 3 products; FP64 alike to 1e-13."""
    sk = gpu_module()
    V = wl.kuhn_vertices(n, 0.16, 3)
    S = sk.Stokes(n, V, 1e-2, 1e-3, 0.0, sk.stokes_default_options(precision=1))
    orc = StokesSystem(KuhnMesh(n, V), 1e-2, 1e-3)
    rng = np.random.default_rng(n)
    u = rng.standard_normal(orc.B.shape[1]).astype(np.float32).astype(np.float64)
    q = rng.standard_normal(orc.B.shape[0]).astype(np.float32).astype(np.float64)
    for suffix, bound in (("", 1e-13), ("_F32", BOUND)):
        bu = host(S.apply("B" + suffix, cuda(soa(u)), q.size))
        btq = aos(host(S.apply("BT" + suffix, cuda(q), u.size)))
        assert np.linalg.norm(bu - orc.B @ u) <= bound * np.linalg.norm(abs(orc.B) @ abs(u))
        assert np.linalg.norm(btq - orc.B.T @ q) <= bound * np.linalg.norm(abs(orc.B.T) @ abs(q))
    S.close()


@pytest.mark.parametrize("n", [4, 5, 7, 8, 12, 33])
def test_fp32_transfers_without_matrices(n):
    """Prolongation (nested and odd meshes) and restriction (nested) in FP32
    against the assembled FP64 transfer matrices, on every level."""
    sk = gpu_module()
    S = sk.Stokes(n, wl.kuhn_vertices(n, 0.1, 1), 1e-2, 1e-3, 0.0, sk.stokes_default_options(precision=1))
    rng = np.random.default_rng(n)
    sizes, m = [], n
    while True:
        sizes.append(3 * (2 * m - 1) ** 3)
        if m < 4:
            break
        m = (m + 1) // 2
    for level in range(len(sizes) - 1):
        for op, nx, ny in (("PROLONG_P2", sizes[level + 1], sizes[level]), ("RESTRICT_P2", sizes[level], sizes[level + 1])):
            x = rng.standard_normal(nx).astype(np.float32).astype(np.float64)
            want = host(S.apply(op, cuda(x), ny, level))
            size = host(S.apply(op, cuda(abs(x)), ny, level))  # (weights of both signs: a lower bound of |P||x|)
            got = host(S.apply(op + "_F32", cuda(x), ny, level))
            assert np.linalg.norm(got - want) <= BOUND * (np.linalg.norm(size) + np.linalg.norm(want))
    S.close()


@pytest.mark.parametrize("n", [3, 16, 17, 26, 33])
def test_stencil_products_across_warp_splits(n):
    """A~_3 and the P1 operators from stencil storage against their exported
    CSR matrices, with level sizes on both sides of the lines where a row's
    entries go over 8, 4, 2 warps or one thread (2^15, 2^17, 2^18 rows); sums
    of up to 65 FP64 products."""
    sk = gpu_module()
    S = sk.Stokes(n, wl.kuhn_vertices(n, 0.16, 5), 1e-2, 1e-3)
    rng = np.random.default_rng(n)
    for op, comps in (("A3", 3), ("KQ", 1), ("MQ", 1), ("LQ", 1)):
        rp, ci, v, shp = S.matrix(op)
        M = to_scipy(rp, ci, v, shp)
        x = rng.standard_normal((comps, shp[1]))
        y = host(S.apply(op, cuda(x.ravel()), comps * shp[0])).reshape(comps, -1)
        for c in range(comps):
            assert np.linalg.norm(y[c] - M @ x[c]) <= 1e-14 * np.linalg.norm(abs(M) @ abs(x[c]))
    S.close()


@pytest.mark.parametrize("n", [5, 9, 13])
def test_fp32_strain_product_of_smooth_vectors(n):
    """Where the mass term dominates, a smooth vector leaves no cancellation to
    hide behind: the error stays below that of the product with the matrix
    blocks rounded to FP32 (4.8e-8, about 0.8 units of rounding)."""
    sk = gpu_module()
    mu = dt = 1e-4
    V = wl.kuhn_vertices(n, 0.16, 7)
    S = sk.Stokes(n, V, mu, dt, 0.0, sk.stokes_default_options(precision=1))
    orc = StokesSystem(KuhnMesh(n, V), mu, dt)
    t = np.arange(1, 2 * n) / (2 * n)
    z, y, x = np.meshgrid(t, t, t, indexing="ij")
    s = np.sin(np.pi * x) * np.sin(np.pi * y) * np.sin(np.pi * z)
    v = np.stack([s, 2 * s * (1 + x), -s * (1.5 + y)], axis=-1).ravel().astype(np.float32).astype(np.float64)
    got = aos(host(S.apply("A_F32", cuda(soa(v)), v.size)))
    want = orc.A @ v
    assert np.linalg.norm(got - want) <= 0.8 * 2.0 ** -24 * np.linalg.norm(want)
    S.close()


@pytest.mark.parametrize("n", [2, 5, 8])
def test_divergence_of_non_finite_entries(n):
    """An infinity in x reaches the rows of B that hold its node and no others
    (rows of other nodes whose offsets leave the mesh alias it in the linear
    index), in one system and in one of four."""
    sk = gpu_module()
    V = wl.kuhn_vertices(n, 0.16, 3)
    S = sk.Stokes(n, V, 1e-2, 1e-3, 0.0, sk.stokes_default_options(precision=1))
    orc = StokesSystem(KuhnMesh(n, V), 1e-2, 1e-3)
    nv, npr = orc.A.shape[0], orc.B.shape[0]
    rng = np.random.default_rng(n)
    u = rng.standard_normal((4, nv)).astype(np.float32).astype(np.float64)
    for node in (0, nv // 6, nv // 3 - 1):  # the first, a middle and the last interior node
        bad = u[0].copy()
        bad[3 * node + 1] = np.inf
        touched = np.asarray(abs(orc.B)[:, 3 * node:3 * node + 3].sum(axis=1)).ravel() > 0
        assert touched.any()
        four = np.stack([soa(u[1]), soa(bad), soa(u[2]), soa(u[3])])
        y4 = host(S.apply("B_F32_X4", cuda(np.concatenate([four.ravel(), np.zeros(4 * npr)])), 4 * npr)).reshape(4, npr)
        finite = host(S.apply("B_F32_X4", cuda(np.concatenate([np.stack([soa(v) for v in u]).ravel(), np.zeros(4 * npr)])),
                              4 * npr)).reshape(4, npr)
        for op, y, good in (("B", None, None), ("B_F32", None, None), ("X4", y4[1], finite[0])):
            if y is None:
                y, good = (host(S.apply(op, cuda(soa(v)), npr)) for v in (bad, u[0]))
            assert np.array_equal(y[~touched], good[~touched])
            assert not np.isfinite(y[touched]).any()
        for k, j in ((0, 1), (2, 2), (3, 3)):
            assert np.array_equal(y4[k], finite[j])
    S.close()


@pytest.mark.parametrize("n", [2, 5, 8])
def test_stencil_products_of_non_finite_entries(n):
    """The same for A~_3 and the P1 operators, against their exported CSR
    matrices."""
    sk = gpu_module()
    S = sk.Stokes(n, wl.kuhn_vertices(n, 0.16, 5), 1e-2, 1e-3)
    rng = np.random.default_rng(n)
    for op, comps in (("A3", 3), ("KQ", 1), ("MQ", 1), ("LQ", 1)):
        rp, ci, v, shp = S.matrix(op)
        M = to_scipy(rp, ci, v, shp)
        x = rng.standard_normal((comps, shp[1]))
        for node in (0, shp[1] // 2, shp[1] - 1):
            bad = x.copy()
            bad[0, node] = np.inf
            y = host(S.apply(op, cuda(bad.ravel()), comps * shp[0])).reshape(comps, -1)
            touched = np.asarray(abs(M)[:, [node]].sum(axis=1)).ravel() > 0
            assert np.isfinite(y[1:]).all() and np.isfinite(y[0][~touched]).all()
            assert not np.isfinite(y[0][touched]).any()
    S.close()
