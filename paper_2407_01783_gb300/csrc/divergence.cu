// Products with the divergence B (P1 rows, interior P2 columns, 1x3 blocks) and
// its transpose in stencil storage. Every pressure vertex meets the same 65 P2
// half-grid offsets (a block outside the velocity space is stored as 0), so no
// column indices are needed, and one array [entry][3][vertex] serves both
// products: the block B(k, i) that B^T needs for velocity node i and vertex k is
// entry (i - k) of vertex k, and consecutive nodes of one parity class meet
// consecutive vertices, so B^T reads the same words coalesced too.
//
// Bound by HBM on large meshes (5.3 TB/s at 96^3), by loads in flight on small ones
// (40% of the DRAM rate at 36^3): 3 x 65 words per vertex (93 MB FP32 at 48^3, 17%
// less than CSR with its indices) and the vectors. Against the CSR products it replaced, us at
// 12^3, 25^3, 33^3, 48^3, 96^3: B 2.4, 4.1, 6.5, 23, 155 (3.1, 5.8, 10.6, 34,
// 210), B^T 2.9, 3.7, 5.6, 19, 153 (2.2, 4.8, 8.4, 30, 212).
#include <algorithm>
#include <utility>

#include "internal.h"

namespace sk {

// Entry e's half-grid offset, in (z, y, x) order. Two nodes of a Kuhn mesh share a
// tetrahedron with a vertex exactly if the offset lies in {0,1,2}^3, {0,-1,-2}^3
// or {-1,0,1}^3 (all three ends of a monotone path around the vertex).
struct DivOffsets {
  signed char d[kDivS][3];
};
__host__ __device__ constexpr DivOffsets div_table() {
  DivOffsets t{};
  int e = 0;
  for (int z = -2; z <= 2; ++z)
    for (int y = -2; y <= 2; ++y)
      for (int x = -2; x <= 2; ++x) {
        const bool up = x >= 0 && y >= 0 && z >= 0, down = x <= 0 && y <= 0 && z <= 0;
        const bool mixed = x * x <= 1 && y * y <= 1 && z * z <= 1;
        if (!(up || down || mixed)) continue;
        t.d[e][0] = (signed char)x;
        t.d[e][1] = (signed char)y;
        t.d[e][2] = (signed char)z;
        ++e;
      }
  return t;
}
template <int E, int K> __device__ constexpr int div_d() {
  constexpr DivOffsets t = div_table();
  return t.d[E][K];
}

__global__ void k_div_fill(int n, DivOffsets t, const int* __restrict__ rp, const int* __restrict__ col, long long nnz,
                           const double* __restrict__ val, double* __restrict__ out) {
  dep_wait();
  const int nv = n + 1, np = nv * nv * nv, m = 2 * n - 1;
  const int r = blockIdx.x * blockDim.x + threadIdx.x, e = blockIdx.y;
  if (r >= np) return;
  const int q[3] = {2 * (r % nv) + t.d[e][0], 2 * ((r / nv) % nv) + t.d[e][1], 2 * (r / (nv * nv)) + t.d[e][2]};
  double w[3] = {0, 0, 0};
  if (min(min(q[0], q[1]), q[2]) >= 1 && max(max(q[0], q[1]), q[2]) <= m) {  // an interior node
    const int c = (q[0] - 1) + m * ((q[1] - 1) + m * (q[2] - 1));
    int lo = rp[r], hi = rp[r + 1];
    const int end = hi;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (col[mid] < c) lo = mid + 1; else hi = mid;
    }
    if (lo < end && col[lo] == c)
      for (int u = 0; u < 3; ++u) w[u] = val[(size_t)u * nnz + lo];
  }
  for (int u = 0; u < 3; ++u) out[(size_t)(3 * e + u) * np + r] = w[u];
}

DivOp* div_from_csr(const Exec& ex, Arena& ar, const StencilTables* st, int n, const Csr& B) {
  constexpr DivOffsets t = div_table();
  signed char d[kDivS][3];
  div_offsets(st, d);
  for (int e = 0; e < kDivS; ++e)
    for (int k = 0; k < 3; ++k) SK_REQUIRE(d[e][k] == t.d[e][k], STOKES_ERR_ARG, "unexpected divergence stencil");
  auto* o = new DivOp();
  o->n = n;
  const int np = (n + 1) * (n + 1) * (n + 1);
  o->v64 = ar.alloc<double>((size_t)3 * kDivS * np);
  launch_dep(k_div_fill, dim3(cdiv(np, 256), kDivS), 256, 0, ex, n, t, B.rowptr, B.col, B.nnz, B.v64, o->v64);
  SK_CHECK_LAUNCH();
  return o;
}

// y = b + alpha B x for K right-hand sides. A block takes 32 vertices, its warp
// w the entries w, w + 8, ... of each: eight times the loads in flight of a
// thread per row, which small meshes need (17 576 rows at 25^3). A vertex knows
// its interior offsets per axis as bits and leaves the other entries out of its
// sum: their weight is 0, but what is read for them is another node's value, which
// may be an infinity.
__host__ __device__ constexpr unsigned div_bit(int axis, int d) { return 1u << (5 * axis + d + 2); }
template <int E, int N, int K, class T> struct DivRow {  // entries E, E + 8, ... (N of them), all loads issued first
  using Seq = std::make_integer_sequence<int, N>;
  static __device__ __forceinline__ void run(const T* __restrict__ v, const T* __restrict__ x, size_t np, size_t xs,
                                             int m, int base, int last, unsigned in, T* acc) {
    T w[N][3];
    int c[N];
    load(Seq(), v, np, m, base, last, w, c);
#pragma unroll
    for (int q = 0; q < K; ++q) {
      T xv[N][3];
#pragma unroll
      for (int t = 0; t < N; ++t)
#pragma unroll
        for (int u = 0; u < 3; ++u) xv[t][u] = x[(size_t)(3 * q + u) * xs + c[t]];
      add(Seq(), in, w, xv, acc + 2 * q);
    }
  }
  template <int... I>
  static __device__ __forceinline__ void load(std::integer_sequence<int, I...>, const T* __restrict__ v, size_t np,
                                              int m, int base, int last, T (*w)[3], int* c) {
    (one<E + 8 * I>(v, np, m, base, last, w[I], c[I]), ...);
  }
  template <int F>
  static __device__ __forceinline__ void one(const T* __restrict__ v, size_t np, int m, int base, int last, T* w,
                                             int& c) {
#pragma unroll
    for (int u = 0; u < 3; ++u) w[u] = v[(size_t)(3 * F + u) * np];
    c = min(max(base + div_d<F, 0>() + m * (div_d<F, 1>() + m * div_d<F, 2>()), 0), last);  // (absent ones: any)
  }
  template <int... I>
  static __device__ __forceinline__ void add(std::integer_sequence<int, I...>, unsigned in, const T (*w)[3],
                                             const T (*xv)[3], T* acc) {
    (sum<E + 8 * I>(in, w[I], xv[I], acc[I % 2]), ...);
  }
  template <int F>
  static __device__ __forceinline__ void sum(unsigned in, const T* w, const T* xv, T& acc) {
    constexpr unsigned need = div_bit(0, div_d<F, 0>()) | div_bit(1, div_d<F, 1>()) | div_bit(2, div_d<F, 2>());
    const T s = w[0] * xv[0] + w[1] * xv[1] + w[2] * xv[2];
    if ((in & need) == need) acc += s;
  }
};
template <int W, int K, class T>
__device__ __forceinline__ void div_warp(int w, const T* __restrict__ v, const T* __restrict__ x, size_t np, size_t xs,
                                         int m, int base, int last, unsigned in, T* acc) {
  if (w == W) {
    constexpr int N = (kDivS - W + 7) / 8;
    constexpr int H = K > 1 || sizeof(T) == 8 ? N / 2 : N;  // (registers: in two parts)
    DivRow<W, H, K, T>::run(v, x, np, xs, m, base, last, in, acc);
    if constexpr (N > H) DivRow<W + 8 * H, N - H, K, T>::run(v, x, np, xs, m, base, last, in, acc);
  } else if constexpr (W < 7) {
    div_warp<W + 1, K, T>(w, v, x, np, xs, m, base, last, in, acc);
  }
}

template <int K, class T>
__global__ void __launch_bounds__(256, 4) k_div(int n, FastDiv by_v, FastDiv by_vv, const T* __restrict__ v,
                                                const T* __restrict__ x, const T* b, T alpha, T* y) {
  dep_wait();
  __shared__ T sh[8][K][32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nv = n + 1, np = nv * nv * nv, m = 2 * n - 1;
  const size_t xs = (size_t)m * m * m;
  const int r = blockIdx.x * 32 + lane, rr = min(r, np - 1);
  const int k = by_vv.div(rr), rk = rr - k * by_vv.d, j = by_v.div(rk), i = rk - j * nv;
  const int base = (2 * i - 1) + m * ((2 * j - 1) + m * (2 * k - 1)), last = (int)xs - 1;
  unsigned in = 0;
#pragma unroll
  for (int d = -2; d <= 2; ++d) {
    const auto inside = [&](int a) { return 2 * a + d >= 1 && 2 * a + d <= m; };
    in |= (inside(i) ? div_bit(0, d) : 0u) | (inside(j) ? div_bit(1, d) : 0u) | (inside(k) ? div_bit(2, d) : 0u);
  }
  T acc[2 * K];  // two partial sums each
#pragma unroll
  for (int q = 0; q < 2 * K; ++q) acc[q] = T(0);
  div_warp<0, K, T>(w, v + rr, x, np, xs, m, base, last, in, acc);
#pragma unroll
  for (int q = 0; q < K; ++q) sh[w][q][lane] = acc[2 * q] + acc[2 * q + 1];
  __syncthreads();
  if (w < K && r < np) {
    const T s = ((sh[0][w][lane] + sh[1][w][lane]) + (sh[2][w][lane] + sh[3][w][lane])) +
                ((sh[4][w][lane] + sh[5][w][lane]) + (sh[6][w][lane] + sh[7][w][lane]));
    const size_t at = (size_t)w * np + r;
    y[at] = b ? b[at] + alpha * s : alpha * s;
  }
}

// y = b + alpha s o (B^T x) for K right-hand sides: a thread per velocity node,
// blockIdx.y its parity class C (bits: odd x, y, z). The vertices that share a
// tetrahedron with a node of the class are the entries of B with that parity.
// (two partial sums, alternating: H picks the one of entry E)
template <int C, int E, int H, int K, class T>
__device__ __forceinline__ void divt_entries(const T* __restrict__ v, const T* __restrict__ x, int np, int nv, int base,
                                             T (*acc)[3 * K]) {
  constexpr int dx = div_d<E, 0>(), dy = div_d<E, 1>(), dz = div_d<E, 2>();
  constexpr bool mine = (dx & 1) == (C & 1) && (dy & 1) == ((C >> 1) & 1) && (dz & 1) == (C >> 2);
  if constexpr (mine) {
    // vertex (q - d) / 2 against q >> 1; every such vertex exists
    const int k = base + ((C & 1) - dx) / 2 + nv * ((((C >> 1) & 1) - dy) / 2 + nv * (((C >> 2) - dz) / 2));
    T w[3];
#pragma unroll
    for (int u = 0; u < 3; ++u) w[u] = v[(size_t)(3 * E + u) * np + k];
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const T xv = x[(size_t)q * np + k];
#pragma unroll
      for (int u = 0; u < 3; ++u) acc[H][3 * q + u] += w[u] * xv;
    }
  }
  if constexpr (E + 1 < kDivS) divt_entries<C, E + 1, mine ? 1 - H : H, K, T>(v, x, np, nv, base, acc);
}
template <int C, int K, class T>
__device__ __forceinline__ void divt_class(int c, const T* __restrict__ v, const T* __restrict__ x, int np, int nv,
                                           int base, T (*acc)[3 * K]) {
  if (c == C) divt_entries<C, 0, 0, K, T>(v, x, np, nv, base, acc);
  else if constexpr (C < 7) divt_class<C + 1, K, T>(c, v, x, np, nv, base, acc);
}

template <int K, class T>
__global__ void __launch_bounds__(256) k_divt(int n, FastDiv by_o, FastDiv by_e, const T* __restrict__ v,
                                              const T* __restrict__ x, const T* __restrict__ scale, const T* b, T alpha,
                                              T* y) {
  dep_wait();
  const int c = blockIdx.y, nv = n + 1, np = nv * nv * nv, m = 2 * n - 1;
  const int odd[3] = {c & 1, (c >> 1) & 1, c >> 2};
  const int ex = n - 1 + odd[0], ey = n - 1 + odd[1], ez = n - 1 + odd[2];
  const int t = blockIdx.x * 256 + threadIdx.x;
  if (t >= ex * ey * ez) return;
  // division by n (odd coordinate) or n - 1
  const int lines = (odd[0] ? by_o : by_e).div(t), kz = (odd[1] ? by_o : by_e).div(lines);
  const int qx = 2 - odd[0] + 2 * (t - lines * ex), qy = 2 - odd[1] + 2 * (lines - kz * ey), qz = 2 - odd[2] + 2 * kz;
  const int base = (qx >> 1) + nv * ((qy >> 1) + nv * (qz >> 1));
  T acc[2][3 * K];
#pragma unroll
  for (int q = 0; q < 3 * K; ++q) acc[0][q] = acc[1][q] = T(0);
  divt_class<0, K, T>(c, v, x, np, nv, base, acc);
  const size_t ns = (size_t)m * m * m;
  const size_t row = (size_t)(qx - 1) + (size_t)m * ((qy - 1) + (size_t)m * (qz - 1));
  const T f = alpha * (scale ? scale[row] : T(1));
#pragma unroll
  for (int q = 0; q < 3 * K; ++q) {
    const size_t at = q * ns + row;
    const T s = f * (acc[0][q] + acc[1][q]);
    y[at] = b ? b[at] + s : s;
  }
}

template <class T>
void div_apply(const Exec& ex, const DivOp& d, int k, const T* x, T* y, const T* b, double alpha) {
  const int np = (d.n + 1) * (d.n + 1) * (d.n + 1);
  const FastDiv by_v(d.n + 1), by_vv((d.n + 1) * (d.n + 1));
  if (k == 4) launch_dep(k_div<4, T>, cdiv(np, 32), 256, 0, ex, d.n, by_v, by_vv, d.template v<T>(), x, b, (T)alpha, y);
  else launch_dep(k_div<1, T>, cdiv(np, 32), 256, 0, ex, d.n, by_v, by_vv, d.template v<T>(), x, b, (T)alpha, y);
  SK_CHECK_LAUNCH();
}
template <class T>
void divt_apply(const Exec& ex, const DivOp& d, int k, const T* x, T* y, const T* scale, const T* b, double alpha) {
  const dim3 grid(cdiv((long long)d.n * d.n * d.n, 256), 8);
  const FastDiv by_o(d.n), by_e(d.n - 1);
  if (k == 4) launch_dep(k_divt<4, T>, grid, 256, 0, ex, d.n, by_o, by_e, d.template v<T>(), x, scale, b, (T)alpha, y);
  else launch_dep(k_divt<1, T>, grid, 256, 0, ex, d.n, by_o, by_e, d.template v<T>(), x, scale, b, (T)alpha, y);
  SK_CHECK_LAUNCH();
}

template void div_apply<float>(const Exec&, const DivOp&, int, const float*, float*, const float*, double);
template void div_apply<double>(const Exec&, const DivOp&, int, const double*, double*, const double*, double);
template void divt_apply<float>(const Exec&, const DivOp&, int, const float*, float*, const float*, const float*,
                                double);
template void divt_apply<double>(const Exec&, const DivOp&, int, const double*, double*, const double*, const double*,
                                 double);

}  // namespace sk
