// FP32 products with the strain-form velocity operator A evaluated element by
// element (matrix-free) from the geometry of the tetrahedra: 10 words per
// tetrahedron instead of the ~170 of the assembled blocks.
//
// On an affine tetrahedron the gradient of a P2 function is linear, so it is
// given by its values at the four vertices k,
//   grad u (k) = sum_m D_m^k g_m,  D_m^k = 3 u_m (k = m), 4 u_mk - u_m (k != m),
// with u_m the vertex values, u_mk the edge values and g_m the barycentric
// gradients, and products of two linear fields integrate exactly as
// |K|/20 sum_kl (1 + delta_kl). The mass term uses the closed-form P2 mass
// matrix (420/|K| times small integers).
//
// Two kernels per product. k_el_strain: a block takes 32 consecutive cubes and
// its warp p their tetrahedra p (a lane per cube); the warps leave the ten
// nodal results of every tetrahedron in shared memory and then add them up per
// node of the cube, the nodes shared by two neighbours along x included, so 18
// instead of 60 words per cube and component go to the work space. k_el_sum: a
// thread per cube and component adds, in a fixed order, the partials of the
// eight nodes that the cube owns (its low corner and the seven half-grid nodes
// above it) and applies the epilogue. No atomics: the result is deterministic.
#include <algorithm>

#include "internal.h"

namespace sk {

// local node numbers (ox + 3 oy + 9 oz in the cube's 3x3x3 half-grid block) of
// the Kuhn tetrahedra: tetrahedron p walks from the low to the high corner along
// the axes of permutation p; vertices 0..3, then edges 01 02 03 12 13 23
__host__ __device__ constexpr int el_axis(int p, int s) {
  constexpr int t[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
  return t[p][s];
}
__host__ __device__ constexpr int el_stride(int axis) { return axis == 0 ? 1 : (axis == 1 ? 3 : 9); }
// half the local number of vertex v (vertex numbers are even multiples)
__host__ __device__ constexpr int el_vertex(int p, int v) {
  int s = 0;
  for (int k = 0; k < v; ++k) s += el_stride(el_axis(p, k));
  return s;
}
__host__ __device__ constexpr int el_edge(int a, int b) {  // index 0..5 of edge ab
  return a == 0 ? b - 1 : (b == 0 ? a - 1 : a + b);
}
__host__ __device__ constexpr int el_end(int e, int s) {  // ends of edge e
  constexpr int t[6][2] = {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}};
  return t[e][s];
}
__host__ __device__ constexpr int el_node(int p, int a) {
  return a < 4 ? 2 * el_vertex(p, a) : el_vertex(p, el_end(a - 4, 0)) + el_vertex(p, el_end(a - 4, 1));
}

// Geometry record of a tetrahedron: kElWords words, 0..8: sqrt(|K|/20) g_m[c] at
// 3 (m - 1) + c, m = 1..3; 9: |K| / (420 dt). Records of tetrahedron p of the 32
// cubes of block q are stored [p][q][word / 4][cube][word % 4], so a warp reads
// them as three coalesced 16-byte loads per lane.
__host__ __device__ __forceinline__ size_t el_blocks(size_t nc) { return (nc + 31) / 32; }
__global__ void k_el_geometry(int n, const double* __restrict__ X, double dt, float* __restrict__ G) {
  dep_wait();
  const size_t nc = (size_t)n * n * n;
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 6 * nc) return;
  const int p = (int)(t / nc);
  const size_t cube = t - p * nc;
  const int i = (int)(cube % n), j = (int)((cube / n) % n), k = (int)(cube / ((size_t)n * n));
  const int nv = n + 1;
  size_t id = (size_t)i + nv * ((size_t)j + (size_t)nv * k);
  double x0[3], e[3][3];
  for (int c = 0; c < 3; ++c) x0[c] = X[3 * id + c];
  for (int s = 0; s < 3; ++s) {
    const int a = el_axis(p, s);
    id += a == 0 ? 1 : (a == 1 ? nv : (size_t)nv * nv);
    for (int c = 0; c < 3; ++c) e[s][c] = X[3 * id + c] - x0[c];
  }
  double g[3][3];
  for (int s = 0; s < 3; ++s) {
    const double* u = e[(s + 1) % 3];
    const double* v = e[(s + 2) % 3];
    for (int c = 0; c < 3; ++c) g[s][c] = u[(c + 1) % 3] * v[(c + 2) % 3] - u[(c + 2) % 3] * v[(c + 1) % 3];
  }
  const double det = e[0][0] * g[0][0] + e[0][1] * g[0][1] + e[0][2] * g[0][2];
  const double vol = fabs(det) / 6.0, w = sqrt(vol / 20.0) / det;
  float* o = G + ((size_t)p * el_blocks(nc) + cube / 32) * (32 * kElWords) + 4 * (cube % 32);
  float r[kElWords] = {};
  for (int s = 0; s < 3; ++s)
    for (int c = 0; c < 3; ++c) r[3 * s + c] = (float)(w * g[s][c]);
  r[9] = (float)(vol / (420.0 * dt));
  for (int q = 0; q < kElWords; ++q) o[128 * (q / 4) + q % 4] = r[q];
}

float* element_geometry(const Exec& ex, Arena& ar, int n, const double* X, double dt) {
  const size_t nc = (size_t)n * n * n;
  float* G = ar.alloc<float>(6 * 32 * kElWords * el_blocks(nc));
  launch_dep(k_el_geometry, cdiv((long long)(6 * nc), 256), 256, 0, ex, n, X, dt, G);
  SK_CHECK_LAUNCH();
  return G;
}

// Nodes of tetrahedron p as seen by one lane: vertex v lies at the cube's low
// corner plus the axes in the bit set C[v], V[v] its index offset in half-grid
// steps; lo and hi are the axes along which the cube touches the boundary.
struct ElNodes {
  int C[4], V[4];
  unsigned lo, hi;
  __device__ __forceinline__ ElNodes(int p, int n, int i, int j, int k) {
    const int a0 = p >> 1, a1 = p == 0 || p == 5 ? 1 : (p == 1 || p == 3 ? 2 : 0);  // el_axis(p, 0), el_axis(p, 1)
    const int m = 2 * n - 1;
    C[0] = 0, C[1] = 1 << a0, C[2] = C[1] | 1 << a1, C[3] = 7;
#pragma unroll
    for (int v = 0; v < 4; ++v) V[v] = (C[v] & 1) + m * (((C[v] >> 1) & 1) + m * (C[v] >> 2));
    lo = (i == 0) | (j == 0) << 1 | (k == 0) << 2;
    hi = (i == n - 1) | (j == n - 1) << 1 | (k == n - 1) << 2;
  }
  // node a (vertices, then edges): offset, and whether it is an interior node
  __device__ __forceinline__ int offset(int a) const {
    return a < 4 ? 2 * V[a] : V[el_end(a - 4, 0)] + V[el_end(a - 4, 1)];
  }
  __device__ __forceinline__ bool inside(int a) const {
    const int c = C[a < 4 ? a : el_end(a - 4, 0)], d = C[a < 4 ? a : el_end(a - 4, 1)];
    return !((lo & ~(c | d)) | (hi & (c & d)));
  }
};

// Strain-form result y (edges: a quarter of it) of one tetrahedron for nodal
// values u (vertices, then edges), geometry g and w; mu the viscosity. Gradients
// and all but the row sums of the mass matrix (-21 and 84 of 420) act on the
// differences to the mean r of the edge values: sums of near-equal numbers and
// their cancellation in the gradients are what costs FP32 its last bits.
__device__ __forceinline__ void el_strain_tet(float (&u)[10][3], float (&y)[10][3], const float (&g)[3][3],
                                              float w, float mu) {
  float H[4][3][3];  // H[k][p][c] = d_p u_c at vertex k (scaled)
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float r =
        (((u[6][c] + u[7][c]) + (u[5][c] + u[8][c])) + (u[4][c] + u[9][c])) * (float)(1.0 / 6.0);
#pragma unroll
    for (int a = 0; a < 10; ++a) u[a][c] -= r;
    float D[4][4];
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int k = 0; k < 4; ++k)
        D[m][k] = m == k ? 3.f * u[m][c] : 4.f * u[4 + el_edge(m, k)][c] - u[m][c];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float d[3];
#pragma unroll
      for (int m = 1; m < 4; ++m) d[m - 1] = D[m][k] - D[0][k];
#pragma unroll
      for (int p = 0; p < 3; ++p) H[k][p][c] = g[0][p] * d[0] + g[1][p] * d[1] + g[2][p] * d[2];
    }
    // mass: vertex i: V + 5 u_i - 6 S + 2 E_i, edge ij: 16 S + 16 u_ij - 8 u_opposite - 6 V + 2 (u_i + u_j)
    // (V, S: sums over vertices and edges, E_i: over the edges at i)
    float E[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      float s = 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k != m) s += u[4 + el_edge(m, k)][c];
      E[m] = s;
    }
    const float S = 0.5f * ((E[0] + E[1]) + (E[2] + E[3]));
    const float V = (u[0][c] + u[1][c]) + (u[2][c] + u[3][c]);
    const float vs = V - 6.f * S, es = 4.f * S - 1.5f * V;
#pragma unroll
    for (int m = 0; m < 4; ++m) y[m][c] = w * (vs + 5.f * u[m][c] + 2.f * E[m] - 21.f * r);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = a + 1; b < 4; ++b) {
        const int e = el_edge(a, b);  // the opposite edge is 5 - e
        y[4 + e][c] = w * (es + 4.f * u[4 + e][c] - 2.f * u[9 - e][c] + 0.5f * (u[a][c] + u[b][c]) + 21.f * r);
      }
  }
  // strain at the vertices, weighted by the P1 mass: T[k] = mu (S[k] + sum_l S[l])
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int c = p; c < 3; ++c) {
      float s[4], t = 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        s[k] = H[k][p][c] + H[k][c][p];
        t += s[k];
      }
      t *= mu;
#pragma unroll
      for (int k = 0; k < 4; ++k) H[k][p][c] = H[k][c][p] = mu * s[k] + t;
    }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float F[4][4];  // F[m][k]
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int m = 1; m < 4; ++m)
        F[m][k] = g[m - 1][0] * H[k][0][c] + g[m - 1][1] * H[k][1][c] + g[m - 1][2] * H[k][2][c];
      F[0][k] = -(F[1][k] + F[2][k] + F[3][k]);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      float s = 3.f * F[m][m];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k != m) s -= F[m][k];
      y[m][c] += s;
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = a + 1; b < 4; ++b) y[4 + el_edge(a, b)][c] += F[a][b] + F[b][a];
  }
}

// Work space, per block of 32 cubes and component kElRows rows of 32 words:
// row 2 (oy + 3 oz) + ox, ox in {0, 1}, holds the cubes' nodes (the node with
// ox = 0 includes its left neighbour's share when both cubes are in the block),
// row 18 at oy + 3 oz the share of the block's last cube in its ox = 2 nodes.
constexpr int kElRows = 19;
__host__ __device__ __forceinline__ size_t el_part_words(size_t nc) { return 3 * 32 * kElRows * el_blocks(nc); }

// sum over the tetrahedra that hold node O of the cube, in order of p
template <int O> __device__ __forceinline__ float el_tet_sum(const float (*sh)[30][32], int c, int lane) {
  float s = 0.f;
#pragma unroll
  for (int p = 0; p < 6; ++p)
#pragma unroll
    for (int a = 0; a < 10; ++a)
      if (el_node(p, a) == O) s += sh[p][3 * a + c][lane];
  return s;
}
template <int Q, int OX>  // Q = oy + 3 oz; part: the block's rows of component c
__device__ __forceinline__ void el_combine(const float (*sh)[30][32], int c, int lane, bool left,
                                           float* __restrict__ part) {
  float s = el_tet_sum<3 * Q + OX>(sh, c, lane);
  if constexpr (OX == 0) {
    const float r = el_tet_sum<3 * Q + 2>(sh, c, lane);
    const float l = __shfl_up_sync(0xffffffffu, r, 1);
    if (left) s += l;
    if (lane == 31) part[32 * 18 + Q] = r;
  }
  part[32 * (2 * Q + OX) + lane] = s;
  if constexpr (Q < 8) el_combine<Q + 1, OX>(sh, c, lane, left, part);
}

constexpr int kElBlock = 192;  // 32 cubes x 6 tetrahedra

// What bounds it: instruction issue (about 700 FP32 operations per tetrahedron,
// half of all instructions), 0.6 warps per clock and scheduler. Four resident
// blocks at 80 registers measured best (3, 4, 5 blocks: 32.4, 30.9, 31.4 us at
// 48^3), one thread per cube with 255 registers 35 us there and 8 us instead of
// 3.4 us on small meshes (one long chain per cube). Product with k_el_sum
// against the symmetric storage it replaced (2.8 TB/s on 446 MB at 48^3):
// 12^3 7.6 us (16), 25^3 11 (31), 33^3 17 (60), 48^3 40 (165), 64^3 87 (352),
// 96^3 289 (1267).
// Error against FP64 over n = 12..96, (mu, dt) from (1e-6, 1e-2) to (1, 1e-2):
// N(0,1) vectors 5.1e-8..6.8e-8 relative (the FP32 blocks: 6.3e-8..7.5e-8);
// smooth vectors 4.3e-8 where the mass dominates (4.8e-8), 2.9e-7 at 96^3, mu = 1
// (1.9e-5). Without the differences to the mean, which cost 0.2 of 45.4 us at
// 48^3 and 1.9 of 290.9 at 96^3 (with events around the launches): 5.5e-8..7.0e-8,
// 5.6e-8, 1.1e-5.
__global__ void __launch_bounds__(kElBlock, 4) k_el_strain(int n, const float* __restrict__ G, float mu,
                                                       const float* __restrict__ x, size_t xs,
                                                       float* __restrict__ part) {
  dep_wait();
  __shared__ float sh[6][30][32];
  const int nc = n * n * n, m = 2 * n - 1;
  const int p = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cube = blockIdx.x * 32 + lane;
  const int cc = min(cube, nc - 1);  // lanes past the end repeat the last cube; k_el_sum does not read them
  const int i = cc % n, j = (cc / n) % n, k = cc / (n * n);
  x += (size_t)blockIdx.y * 3 * xs;
  part += ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * (3 * 32 * kElRows);
  {
    const int base = (2 * i - 1) + m * ((2 * j - 1) + m * (2 * k - 1));
    const ElNodes nd(__shfl_sync(0xffffffffu, p, 0), n, i, j, k);
    float g[3][3], w, u[10][3], y[10][3];
    const float4* Gp = reinterpret_cast<const float4*>(G) + ((size_t)p * gridDim.x + blockIdx.x) * (8 * kElWords) + lane;
    const float4 g0 = Gp[0], g1 = Gp[32];
    const float2 g2 = *reinterpret_cast<const float2*>(Gp + 64);
    g[0][0] = g0.x, g[0][1] = g0.y, g[0][2] = g0.z, g[1][0] = g0.w;
    g[1][1] = g1.x, g[1][2] = g1.y, g[2][0] = g1.z, g[2][1] = g1.w;
    g[2][2] = g2.x, w = g2.y;
#pragma unroll
    for (int a = 0; a < 10; ++a) {
      const bool in = nd.inside(a);  // else a boundary node: value 0
      const int at = base + nd.offset(a);
#pragma unroll
      for (int c = 0; c < 3; ++c) u[a][c] = in ? x[c * xs + at] : 0.f;
    }
    el_strain_tet(u, y, g, w, mu);
#pragma unroll
    for (int a = 0; a < 10; ++a)
#pragma unroll
      for (int c = 0; c < 3; ++c) sh[p][3 * a + c][lane] = y[a][c];
  }
  __syncthreads();
  const int c = p % 3;
  part += 32 * kElRows * c;
  if (p < 3) el_combine<0, 1>(sh, c, lane, false, part);
  else el_combine<0, 0>(sh, c, lane, lane > 0 && i > 0, part);
}

// sums of the partials of the eight nodes that cube (i, j, k) owns:
// node 2 (i, j, k) + (a, b, d), a, b, d in {0, 1}; an even coordinate is shared
// with the cube before along that axis. `part` points at the component's
// work space. Nodes with an even coordinate 0 are boundary nodes (not stored).
struct ElNear {  // rows of the cubes (i, j, k), (i, j - 1, k), (i, j, k - 1), (i, j - 1, k - 1)
  const float* p[4];
  bool first[4];  // first of its block
};
template <int A, int B, int D> __device__ __forceinline__ float el_node_sum(const ElNear& e) {
  float s = 0.f;
#pragma unroll
  for (int dz = 0; dz <= 1 - D; ++dz)
#pragma unroll
    for (int dy = 0; dy <= 1 - B; ++dy) {
      const int q = (B ? 1 : 2 * dy) + 3 * (D ? 1 : 2 * dz), w = dy + 2 * dz;
      s += e.p[w][32 * (2 * q + A)];
      if (A == 0 && e.first[w]) s += e.p[w][32 * 18 + q - 3 * 32 * kElRows];  // the block before
    }
  return (A || B || D) ? 4.f * s : s;
}

// y = A x (b null) or b - A x on one component; dot: += x . (A x) as a
// double-float sum
struct ElOut {
  const float* x;
  const float* b;
  float* y;
  DF s;
  template <bool DOT> __device__ __forceinline__ void put(size_t at, float v) {
    if (DOT) df_dot(s, v, x[at]);
    y[at] = b ? b[at] - v : v;
  }
};

// blocks of one component are contiguous: component c owns blocks
// [c nb, (c + 1) nb); blockIdx.y is the right-hand side
template <bool DOT>
__global__ void __launch_bounds__(256) k_el_sum(int n, int nb, const float* __restrict__ part,
                                               const float* __restrict__ x, size_t xs, const float* __restrict__ b,
                                               float* __restrict__ y, double* partial, unsigned* counter,
                                               double* dot) {
  dep_wait();
  const int nc = n * n * n, m = 2 * n - 1;
  const int c = blockIdx.x / nb;
  const int cube = (blockIdx.x - c * nb) * 256 + threadIdx.x;
  const size_t off = (3 * blockIdx.y + c) * xs;
  ElOut o{x + off, b ? b + off : nullptr, y + off, DF{0.f, 0.f}};
  if (cube < nc) {
    const int i = cube % n, j = (cube / n) % n, k = cube / (n * n);
    const size_t at = (size_t)(2 * i) + (size_t)m * (2 * j + (size_t)m * (2 * k));  // node (1, 1, 1) of the cube
    const size_t my = m, mz = (size_t)m * m;
    const float* pc = part + blockIdx.y * el_part_words(nc) + c * (32 * kElRows);
    ElNear e;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int cw = max(cube - n * ((w & 1) + n * (w >> 1)), 0);  // (absent neighbours are not read)
      e.p[w] = pc + (size_t)(cw >> 5) * (3 * 32 * kElRows) + (cw & 31);
      e.first[w] = (cw & 31) == 0;
    }
    o.put<DOT>(at, el_node_sum<1, 1, 1>(e));
    if (i) o.put<DOT>(at - 1, el_node_sum<0, 1, 1>(e));
    if (j) {
      o.put<DOT>(at - my, el_node_sum<1, 0, 1>(e));
      if (i) o.put<DOT>(at - my - 1, el_node_sum<0, 0, 1>(e));
    }
    if (k) {
      o.put<DOT>(at - mz, el_node_sum<1, 1, 0>(e));
      if (i) o.put<DOT>(at - mz - 1, el_node_sum<0, 1, 0>(e));
      if (j) {
        o.put<DOT>(at - mz - my, el_node_sum<1, 0, 0>(e));
        if (i) o.put<DOT>(at - mz - my - 1, el_node_sum<0, 0, 0>(e));
      }
    }
  }
  if (DOT)
    grid_sum(o.s, partial + (size_t)blockIdx.y * gridDim.x, counter + blockIdx.y, dot + blockIdx.y);
}

size_t element_part_words(int n) { return el_part_words((size_t)n * n * n); }
int element_dot_grid(int n) { return kFusedDots * 3 * cdiv((long long)n * n * n, 256); }

void element_strain(const Exec& ex, const ElementOp& e, int k, const float* x, float* y, const float* b,
                    const DotScratch* ds, double* dot) {
  const int n = e.n, nc = n * n * n;
  const size_t xs = (size_t)(2 * n - 1) * (2 * n - 1) * (2 * n - 1);
  const int nb = cdiv(nc, 256);
  SK_REQUIRE(!dot || (ds && ds->fused_partial && element_dot_grid(n) <= ds->fused_cap), STOKES_ERR_ARG,
             "fused dot scratch too small");
  for (int k0 = 0; k0 < k; k0 += e.batch) {
    const int kk = std::min(e.batch, k - k0);
    const size_t o = (size_t)3 * k0 * xs;
    launch_dep(k_el_strain, dim3(cdiv(nc, 32), kk), kElBlock, 0, ex, n, e.G, e.mu, x + o, xs, e.part);
    SK_CHECK_LAUNCH();
    const dim3 grid(3 * nb, kk);
    if (dot)
      launch_dep(k_el_sum<true>, grid, 256, 0, ex, n, nb, e.part, x + o, xs, b ? b + o : nullptr, y + o, ds->fused_partial,
                                             ds->fused_counter, dot + k0);
    else
      launch_dep(k_el_sum<false>, grid, 256, 0, ex, n, nb, e.part, x + o, xs, b ? b + o : nullptr, y + o, nullptr, nullptr,
                                              nullptr);
    SK_CHECK_LAUNCH();
  }
}

}  // namespace sk
