// Sparse products for the Stokes operators: vectorised CSR (G threads per row,
// shuffle reduction inside the group) over scalar, 3x3, 1x3 and 3x1 blocks,
// with fused epilogues (store, residual, accumulate, Chebyshev update, row
// scaling). All of it is HBM-bound: the matrix is streamed once per product
// (coalesced, values stored as planes of nnz entries), the gathered vector
// mostly hits L2. The number of threads per row is picked per matrix by a
// timing sweep at setup.
#include <dlfcn.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <string>

#include "internal.h"

namespace sk {

// ---------------------------------------------------------------------------
// profiling helpers
// ---------------------------------------------------------------------------
cudaEvent_t Prof::get() {
  if (!pool.empty()) {
    cudaEvent_t e = pool.back();
    pool.pop_back();
    return e;
  }
  cudaEvent_t e;
  SK_CUDA(cudaEventCreate(&e));
  return e;
}

void Prof::reset() {
  for (auto& r : rec) {
    for (auto& p : r.ev) {
      pool.push_back(p.first);
      pool.push_back(p.second);
    }
    r.ev.clear();
    r.bytes = 0;
    r.launches = 0;
    r.ev_bytes = 0;
    r.ev_launches = 0;
  }
}

Prof::~Prof() {
  reset();
  for (auto e : pool) cudaEventDestroy(e);
}

ProfScope::ProfScope(const Exec& e, int k, double bytes) : ex(e), kind(k) {
  if (ex.prof && ex.prof->capture && kind >= 0) {
    ex.prof->capture->bytes[kind] += bytes;
    ex.prof->capture->launches[kind] += 1;
    return;
  }
  if (ex.prof && ex.prof->on && kind >= 0) {
    ex.prof->rec[kind].bytes += bytes;
    ex.prof->rec[kind].launches += 1;
    if (ex.prof->only < 0 || ex.prof->only == kind) {
      e1 = ex.prof->get();
      cudaEventRecord(e1, ex.s);
      ex.prof->rec[kind].ev_bytes += bytes;
      ex.prof->rec[kind].ev_launches += 1;
    }
  }
}

ProfScope::~ProfScope() {
  if (e1) {
    cudaEvent_t e2 = ex.prof->get();
    cudaEventRecord(e2, ex.s);
    ex.prof->rec[kind].ev.emplace_back(e1, e2);
  }
}

// ---------------------------------------------------------------------------
// epilogues: called by lane 0 of each row group with the row sums
// ---------------------------------------------------------------------------
// Vectors with NR components are component-major: component r of row i at
// r * ns + i (ns = number of rows of the vector).
template <class T, int NR> struct EpiStore {
  static constexpr int nr = NR;
  static constexpr bool il = false;
  T* y;
  size_t ns;
  __device__ __forceinline__ void comp(int row, int r, T v) const { y[r * ns + row] = v; }
  __device__ __forceinline__ void operator()(int row, const T* acc) const {
#pragma unroll
    for (int r = 0; r < NR; ++r) comp(row, r, acc[r]);
  }
};
template <class T, int NR> struct EpiAdd {
  static constexpr int nr = NR;
  static constexpr bool il = false;
  T* y;
  size_t ns;
  __device__ __forceinline__ void comp(int row, int r, T v) const { y[r * ns + row] += v; }
  __device__ __forceinline__ void operator()(int row, const T* acc) const {
#pragma unroll
    for (int r = 0; r < NR; ++r) comp(row, r, acc[r]);
  }
};
template <class T, int NR> struct EpiResid {
  static constexpr int nr = NR;
  static constexpr bool il = false;  // y = b - acc
  const T* b;
  T* y;
  size_t ns;
  __device__ __forceinline__ void comp(int row, int r, T v) const { y[r * ns + row] = b[r * ns + row] - v; }
  __device__ __forceinline__ void operator()(int row, const T* acc) const {
#pragma unroll
    for (int r = 0; r < NR; ++r) comp(row, r, acc[r]);
  }
};
template <class T, int NR> struct EpiAxpy {
  static constexpr int nr = NR;
  static constexpr bool il = false;  // y = (b ? b : 0) + alpha * s_row * acc
  const T* b;
  const T* s;
  T* y;
  T alpha;
  size_t ns;
  __device__ __forceinline__ void operator()(int row, const T* acc) const {
    T sc = s ? s[row] : T(1);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      T v = alpha * sc * acc[r];
      if (b) v += b[r * ns + row];
      y[r * ns + row] = v;
    }
  }
};
// Chebyshev semi-iteration step (Saad, Iterative Methods, Alg. 12.1):
// r = b - A x_in; d = c1 d + c2 D^{-1} r; x_out = x_in + d.
template <class T, int NR> struct EpiCheb {
  static constexpr int nr = NR;
  static constexpr bool il = false;
  const T* b;
  const T* xin;
  T* d;
  T* xout;
  const T* dinv;
  T c1, c2;
  size_t ns;
  __device__ __forceinline__ void comp(int row, int r, T v) const {
    const size_t i = r * ns + row;
    const T res = b[i] - v;
    const T dn = c1 * d[i] + c2 * dinv[row] * res;
    d[i] = dn;
    xout[i] = xin[i] + dn;
  }
  __device__ __forceinline__ void operator()(int row, const T* acc) const {
#pragma unroll
    for (int r = 0; r < NR; ++r) comp(row, r, acc[r]);
  }
};

// Same step with a diagonal per component (3x3-block operators): dinv[r*ns+row]
template <class T> struct EpiCheb3 {
  static constexpr int nr = 3;
  static constexpr bool il = false;
  const T* b;
  const T* xin;
  T* d;
  T* xout;
  const T* dinv;
  T c1, c2;
  size_t ns;
  __device__ __forceinline__ void operator()(int row, const T* acc) const {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      size_t i = r * ns + row;
      T res = b[i] - acc[r];
      T dn = c1 * d[i] + c2 * dinv[i] * res;
      d[i] = dn;
      xout[i] = xin[i] + dn;
    }
  }
};

// Node-interleaved vectors (the V-cycles of several right-hand sides):
// component r of row i at i * NR + r, so one row's NR values are contiguous
// and move as 16-byte vectors (NR a multiple of 4 for FP32, of 2 for FP64).
template <class T, int NR> __device__ __forceinline__ void ldv(const T* __restrict__ p, T* o) {
  if constexpr (std::is_same<T, float>::value && NR % 4 == 0) {
#pragma unroll
    for (int i = 0; i < NR / 4; ++i) {
      const float4 v = reinterpret_cast<const float4*>(p)[i];
      o[4 * i] = v.x, o[4 * i + 1] = v.y, o[4 * i + 2] = v.z, o[4 * i + 3] = v.w;
    }
  } else if constexpr (std::is_same<T, double>::value && NR % 2 == 0) {
#pragma unroll
    for (int i = 0; i < NR / 2; ++i) {
      const double2 v = reinterpret_cast<const double2*>(p)[i];
      o[2 * i] = v.x, o[2 * i + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < NR; ++i) o[i] = p[i];
  }
}
template <class T, int NR> __device__ __forceinline__ void stv(T* __restrict__ p, const T* o) {
  if constexpr (std::is_same<T, float>::value && NR % 4 == 0) {
#pragma unroll
    for (int i = 0; i < NR / 4; ++i)
      reinterpret_cast<float4*>(p)[i] = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
  } else if constexpr (std::is_same<T, double>::value && NR % 2 == 0) {
#pragma unroll
    for (int i = 0; i < NR / 2; ++i) reinterpret_cast<double2*>(p)[i] = make_double2(o[2 * i], o[2 * i + 1]);
  } else {
#pragma unroll
    for (int i = 0; i < NR; ++i) p[i] = o[i];
  }
}
template <class T, int NR> struct EpiStoreIL {
  static constexpr int nr = NR;
  static constexpr bool il = true;
  T* y;
  __device__ __forceinline__ void operator()(int row, const T* acc) const { stv<T, NR>(y + (size_t)row * NR, acc); }
};
template <class T, int NR> struct EpiAddIL {
  static constexpr int nr = NR;
  static constexpr bool il = true;
  T* y;
  __device__ __forceinline__ void operator()(int row, const T* acc) const {
    T v[NR];
    ldv<T, NR>(y + (size_t)row * NR, v);
#pragma unroll
    for (int r = 0; r < NR; ++r) v[r] += acc[r];
    stv<T, NR>(y + (size_t)row * NR, v);
  }
};
template <class T, int NR> struct EpiResidIL {
  static constexpr int nr = NR;
  static constexpr bool il = true;
  const T* b;
  T* y;
  __device__ __forceinline__ void operator()(int row, const T* acc) const {
    T v[NR];
    ldv<T, NR>(b + (size_t)row * NR, v);
#pragma unroll
    for (int r = 0; r < NR; ++r) v[r] -= acc[r];
    stv<T, NR>(y + (size_t)row * NR, v);
  }
};
template <class T, int NR> struct EpiChebIL {
  static constexpr int nr = NR;
  static constexpr bool il = true;
  const T* b;
  const T* xin;
  T* d;
  T* xout;
  const T* dinv;
  T c1, c2;
  __device__ __forceinline__ void operator()(int row, const T* acc) const {
    const T di = dinv[row];
    const size_t o = (size_t)row * NR;
    T bv[NR], dv[NR], xv[NR];
    ldv<T, NR>(b + o, bv);
    ldv<T, NR>(d + o, dv);
    ldv<T, NR>(xin + o, xv);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const T dn = c1 * dv[r] + c2 * di * (bv[r] - acc[r]);
      dv[r] = dn;
      xv[r] += dn;
    }
    stv<T, NR>(d + o, dv);
    stv<T, NR>(xout + o, xv);
  }
};

// First two Chebyshev steps from x = 0 in one sweep (node-interleaved): the
// kernel gathers b, and every gathered value is scaled by s0 D^-1 at its
// column, which is the first iterate x1 = d1 = s0 D^-1 b; the epilogue then
// takes the second step r = b - A x1, d = c1 d1 + c2 D^-1 r, x2 = x1 + d.
template <class T, int NR> struct EpiChebFirstIL {
  static constexpr int nr = NR;
  static constexpr bool il = true;
  static constexpr bool first = true;
  const T* b;
  T* d;
  T* xout;
  const T* dinv;
  T s0, c1, c2;
  __device__ __forceinline__ T gather_scale(size_t col) const { return s0 * dinv[col]; }
  __device__ __forceinline__ void operator()(int row, const T* acc) const {
    const T di = dinv[row];
    const size_t o = (size_t)row * NR;
    T bv[NR], dv[NR];
    ldv<T, NR>(b + o, bv);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const T x1 = s0 * di * bv[r];
      const T dn = c1 * x1 + c2 * di * (bv[r] - acc[r]);
      dv[r] = dn;
      bv[r] = x1 + dn;
    }
    stv<T, NR>(d + o, dv);
    stv<T, NR>(xout + o, bv);
  }
};
// the same on component-major vectors
template <class T, int NR> struct EpiChebFirst {
  static constexpr int nr = NR;
  static constexpr bool il = false;
  static constexpr bool first = true;
  const T* b;
  T* d;
  T* xout;
  const T* dinv;
  T s0, c1, c2;
  size_t ns;
  __device__ __forceinline__ T gather_scale(size_t col) const { return s0 * dinv[col]; }
  __device__ __forceinline__ void comp(int row, int r, T v) const {
    const T di = dinv[row];
    const size_t i = r * ns + row;
    const T bv = b[i];
    const T x1 = s0 * di * bv;
    const T dn = c1 * x1 + c2 * di * (bv - v);
    d[i] = dn;
    xout[i] = x1 + dn;
  }
  __device__ __forceinline__ void operator()(int row, const T* acc) const {
#pragma unroll
    for (int r = 0; r < NR; ++r) comp(row, r, acc[r]);
  }
};
template <class E, class = void> struct is_first : std::false_type {};
template <class E> struct is_first<E, std::void_t<decltype(E::first)>> : std::integral_constant<bool, E::first> {};

// Column / row renumbering around another epilogue (the transfers next to a
// parity-split finest level): WithColMap maps every column index the kernel
// reads through sm before the gather; WithRowMap stores row i's result at
// row sm(i).
template <class E> struct WithColMap : E {
  SplitMap sm;
  static constexpr bool colmap = true;
};
template <class E> struct WithRowMap : E {
  SplitMap sm;
  __device__ __forceinline__ void operator()(int row, const typename std::remove_pointer<decltype(E::y)>::type* acc)
      const {
    E::operator()(sm(row), acc);
  }
};
template <class E, class = void> struct has_colmap : std::false_type {};
template <class E> struct has_colmap<E, std::void_t<decltype(E::colmap)>> : std::integral_constant<bool, E::colmap> {};

template <int G, class T, int NR>
__device__ __forceinline__ void group_reduce(T* acc) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1)
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
}

// Batched loads: each lane first issues U independent (column, value) loads of
// its row group (entries k, k+G, ..., k+(U-1)G), then the U gathers of x, then
// the FMAs. One HBM round trip then covers U entries per lane, which is what
// keeps enough bytes in flight per SM to approach the HBM roofline (one
// 4-byte load per lane per round trip is latency-bound at ~35% of peak).
template <int G> struct Batch {
  static constexpr int U = G >= 32 ? 1 : (G >= 16 ? 2 : (G >= 8 ? 4 : 8));
};

// scalar CSR, NR interleaved right-hand sides
template <int G, int NR, class TM, class T, class Epi>
__global__ void __launch_bounds__(256) k_csr(int rows, const int* __restrict__ rp, const int* __restrict__ col,
                                             const TM* __restrict__ val, const T* __restrict__ x, size_t xs,
                                             Epi epi) {
  dep_wait();
  constexpr int U = Batch<G>::U;
  int gt = blockIdx.x * blockDim.x + threadIdx.x;
  int row = gt / G, lane = gt & (G - 1);
  T acc[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) acc[r] = T(0);
  if (row < rows) {
    const int e = rp[row + 1];
    for (int k = rp[row] + lane; k < e; k += U * G) {
      int c[U];
      T a[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        // entries past the row end re-read the row's last entry (always a valid
        // address inside the loop) and contribute zero
        const int kk = k + u * G;
        const bool ok = kk < e;
        const int ks = ok ? kk : e - 1;
        c[u] = col[ks];
        if constexpr (has_colmap<Epi>::value) c[u] = epi.sm(c[u]);
        const T av = (T)val[ks];
        a[u] = ok ? av : T(0);
      }
      T xv[U][NR];
      if constexpr (Epi::il) {
#pragma unroll
        for (int u = 0; u < U; ++u) ldv<T, NR>(x + (size_t)c[u] * NR, xv[u]);
        if constexpr (is_first<Epi>::value) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const T f = epi.gather_scale(c[u]);
#pragma unroll
            for (int r = 0; r < NR; ++r) xv[u][r] *= f;
          }
        }
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int r = 0; r < NR; ++r) xv[u][r] = x[r * xs + c[u]];
        if constexpr (is_first<Epi>::value) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const T f = epi.gather_scale(c[u]);
#pragma unroll
            for (int r = 0; r < NR; ++r) xv[u][r] *= f;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[r] += a[u] * xv[u][r];
    }
  }
  group_reduce<G, T, NR>(acc);
  if (row < rows && lane == 0) epi(row, acc);
}

// 3x3 blocks (strain-form A), planes v[(3c+d)*nnz + k]
template <int G, class T, class Epi>
__global__ void __launch_bounds__(256) k_bsr3(int rows, const int* __restrict__ rp, const int* __restrict__ col,
                                              const T* __restrict__ v, long long nnz, const T* __restrict__ x,
                                              size_t xs, Epi epi) {
  dep_wait();
  constexpr int U = Batch<G>::U > 4 ? 4 : Batch<G>::U;
  int gt = blockIdx.x * blockDim.x + threadIdx.x;
  int row = gt / G, lane = gt & (G - 1);
  T acc[3] = {T(0), T(0), T(0)};
  if (row < rows) {
    const int e = rp[row + 1];
    for (int k = rp[row] + lane; k < e; k += U * G) {
      int c[U];
      T a[U][9];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int kk = k + u * G;
        const bool ok = kk < e;
        const int ks = ok ? kk : e - 1;  // in-bounds re-read, zero contribution
        c[u] = col[ks];
#pragma unroll
        for (int j = 0; j < 9; ++j) {
          const T av = v[(size_t)j * nnz + ks];
          a[u][j] = ok ? av : T(0);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const T x0 = x[c[u]], x1 = x[xs + c[u]], x2 = x[2 * xs + c[u]];
#pragma unroll
        for (int r = 0; r < 3; ++r) acc[r] += a[u][3 * r] * x0 + a[u][3 * r + 1] * x1 + a[u][3 * r + 2] * x2;
      }
    }
  }
  group_reduce<G, T, 3>(acc);
  if (row < rows && lane == 0) epi(row, acc);
}

template <int G>
__global__ void __launch_bounds__(256) k_bsr3_df(int rows, const int* __restrict__ rp, const int* __restrict__ col,
                                                 const float* __restrict__ vh, const float* __restrict__ vl,
                                                 long long nnz, const float* __restrict__ xh,
                                                 const float* __restrict__ xl, size_t xs,
                                                 const double* __restrict__ b, double* __restrict__ y) {
  dep_wait();
  constexpr int U = 2;
  int gt = blockIdx.x * blockDim.x + threadIdx.x;
  int row = gt / G, lane = gt & (G - 1);
  DF acc[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
  if (row < rows) {
    const int e = rp[row + 1];
    for (int k = rp[row] + lane; k < e; k += U * G) {
      int c[U];
      float ah[U][9], al[U][9];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int kk = k + u * G;
        const bool ok = kk < e;
        const int ks = ok ? kk : e - 1;  // in-bounds re-read, zero contribution
        c[u] = col[ks];
#pragma unroll
        for (int j = 0; j < 9; ++j) {
          const float h = vh[(size_t)j * nnz + ks], l = vl[(size_t)j * nnz + ks];
          ah[u][j] = ok ? h : 0.f;
          al[u][j] = ok ? l : 0.f;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        float x_h[3], x_l[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          x_h[q] = xh[q * xs + c[u]];
          x_l[q] = xl[q * xs + c[u]];
        }
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
          for (int q = 0; q < 3; ++q) df_madd(acc[r], ah[u][3 * r + q], al[u][3 * r + q], x_h[q], x_l[q]);
      }
    }
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1)
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const float oh = __shfl_xor_sync(0xffffffffu, acc[r].h, o);
      const float ol = __shfl_xor_sync(0xffffffffu, acc[r].l, o);
      df_add(acc[r], oh, ol);
    }
  if (row < rows && lane == 0) {
    const size_t ns = (size_t)rows;
#pragma unroll
    for (int r = 0; r < 3; ++r) y[r * ns + row] = b[r * ns + row] - ((double)acc[r].h + (double)acc[r].l);
  }
}

template <int G>
static void launch_bsr3_df(const Exec& ex, const Csr& m, const float* xh, const float* xl, const double* b,
                           double* y) {
  const int bs = 256;
  const int grid = cdiv((long long)m.rows * G, bs);
  if (grid == 0) return;
  launch_dep(k_bsr3_df<G>, grid, bs, 0, ex, m.rows, m.rowptr, m.col, m.v32, m.v32lo, m.nnz, xh, xl, m.cols, b, y);
  SK_CHECK_LAUNCH();
}

void bsr3_residual_df(const Exec& ex, const Csr& m, const float* xh, const float* xl, const double* b, double* y,
                      int kind) {
  if (m.sym && m.sym->v32 && m.sym->v32lo) {
    // hi and lo values once, x hi and lo gathered once, b read, y written
    ProfScope ps(ex, kind, (double)m.sym->total * 8.0 + 8.0 * 3 * m.rows + 16.0 * 3 * m.rows);
    sym3_residual_df(ex, m, xh, xl, b, y);
    return;
  }
  SK_REQUIRE(m.v32 && m.v32lo && m.br == 3 && m.bc == 3, STOKES_ERR_ARG, "double-float residual needs A hi/lo");
  // matrix hi+lo planes, column indices, x hi+lo gathered once, b read, y written
  ProfScope ps(ex, kind, (double)m.nnz * (4.0 + 8.0 * 9) + 4.0 * (m.rows + 1) + 8.0 * 3 * m.cols +
                             16.0 * 3 * m.rows);
  switch (m.group) {
    case 1: launch_bsr3_df<1>(ex, m, xh, xl, b, y); break;
    case 2: launch_bsr3_df<2>(ex, m, xh, xl, b, y); break;
    case 4: launch_bsr3_df<4>(ex, m, xh, xl, b, y); break;
    case 8: launch_bsr3_df<8>(ex, m, xh, xl, b, y); break;
    case 16: launch_bsr3_df<16>(ex, m, xh, xl, b, y); break;
    default: launch_bsr3_df<32>(ex, m, xh, xl, b, y); break;
  }
}

// y = A x with 3x3 blocks and *dot = x . y (own-row components of x), the dot
// reduced over the grid in a fixed order (grid_sum); every thread reaches it
template <int G, class T>
__global__ void __launch_bounds__(256) k_bsr3_dot(int rows, const int* __restrict__ rp, const int* __restrict__ col,
                                                  const T* __restrict__ v, long long nnz, const T* __restrict__ x,
                                                  size_t xs, T* __restrict__ y, double* partial, unsigned* counter,
                                                  double* dot) {
  dep_wait();
  constexpr int U = Batch<G>::U > 4 ? 4 : Batch<G>::U;
  // a grid of one resident wave walks the row groups (grid stride), so the
  // grid sum below takes one counter increment per resident block, not per
  // row group
  const int lane = threadIdx.x & (G - 1);
  const int groups = (int)(((long long)rows * G + blockDim.x - 1) / blockDim.x);
  double part = 0.0;
  for (int gb = blockIdx.x; gb < groups; gb += gridDim.x) {
    const int row = (gb * (int)blockDim.x + (int)threadIdx.x) / G;
    T acc[3] = {T(0), T(0), T(0)};
    if (row < rows) {
      const int e = rp[row + 1];
      for (int k = rp[row] + lane; k < e; k += U * G) {
        int c[U];
        T a[U][9];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int kk = k + u * G;
          const bool ok = kk < e;
          const int ks = ok ? kk : e - 1;  // in-bounds re-read, zero contribution
          c[u] = col[ks];
#pragma unroll
          for (int j = 0; j < 9; ++j) {
            const T av = v[(size_t)j * nnz + ks];
            a[u][j] = ok ? av : T(0);
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const T x0 = x[c[u]], x1 = x[xs + c[u]], x2 = x[2 * xs + c[u]];
#pragma unroll
          for (int r = 0; r < 3; ++r) acc[r] += a[u][3 * r] * x0 + a[u][3 * r + 1] * x1 + a[u][3 * r + 2] * x2;
        }
      }
    }
    group_reduce<G, T, 3>(acc);
    if (row < rows && lane == 0) {
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const size_t i = r * xs + row;
        y[i] = acc[r];
        part += (double)(acc[r] * x[i]);
      }
    }
  }
  grid_sum(part, partial, counter, dot);
}

// one resident wave of a kernel: SMs x resident blocks per SM (at most `want`)
template <class K> static int resident_grid(K kernel, int block, int want) {
  int dev = 0, sms = 0, occ = 0;
  SK_CUDA(cudaGetDevice(&dev));
  SK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  SK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, block, 0));
  return std::max(1, std::min(want, sms * std::max(1, occ)));
}

template <int G, class T>
static void launch_bsr3_dot(const Exec& ex, const Csr& m, const T* x, T* y, const DotScratch& ds, double* dot) {
  const int want = cdiv((long long)m.rows * G, 256);
  if (want == 0) return;
  static thread_local int cached[2][6] = {};  // resident wave per (precision, group width)
  int& slot = cached[sizeof(T) == 4][__builtin_ctz(G)];
  if (!slot) slot = resident_grid(k_bsr3_dot<G, T>, 256, 1 << 30);
  const int grid = std::min(want, slot);
  SK_REQUIRE(ds.fused_partial && grid <= ds.fused_cap, STOKES_ERR_ARG, "fused dot scratch too small");
  launch_dep(k_bsr3_dot<G, T>, grid, 256, 0, ex, m.rows, m.rowptr, m.col, m.template v<T>(), m.nnz, x, (size_t)m.cols, y,
                                           ds.fused_partial, ds.fused_counter, dot);
  SK_CHECK_LAUNCH();
}

// upper bound on the blocks of a dot-fused BSR3 launch (one resident wave of
// 256-thread blocks: at most 8 per SM)
int bsr3_dot_grid(const Csr& m) {
  int dev = 0, sms = 0;
  SK_CUDA(cudaGetDevice(&dev));
  SK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  return std::min(cdiv((long long)m.rows * 32, 256), 8 * sms);
}

// 1x3 blocks: B (P1 rows, interior P2 node columns), for K right-hand sides
// (x: 3K component-major components, y: K); the matrix is read once for all
template <int G, int K, class T, class Epi>
__global__ void __launch_bounds__(256) k_b(int rows, const int* __restrict__ rp, const int* __restrict__ col,
                                           const T* __restrict__ v, long long nnz, const T* __restrict__ x, size_t xs,
                                           Epi epi) {
  dep_wait();
  constexpr int U = Batch<G>::U;
  int gt = blockIdx.x * blockDim.x + threadIdx.x;
  int row = gt / G, lane = gt & (G - 1);
  T acc[K];
#pragma unroll
  for (int q = 0; q < K; ++q) acc[q] = T(0);
  if (row < rows) {
    const int e = rp[row + 1];
    for (int k = rp[row] + lane; k < e; k += U * G) {
      int c[U];
      T a[U][3];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int kk = k + u * G;
        const bool ok = kk < e;
        const int ks = ok ? kk : e - 1;  // in-bounds re-read, zero contribution
        c[u] = col[ks];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const T av = v[(size_t)j * nnz + ks];
          a[u][j] = ok ? av : T(0);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int q = 0; q < K; ++q) {
          const T* xq = x + (size_t)3 * q * xs;
          acc[q] += a[u][0] * xq[c[u]] + a[u][1] * xq[xs + c[u]] + a[u][2] * xq[2 * xs + c[u]];
        }
    }
  }
  group_reduce<G, T, K>(acc);
  if (row < rows && lane == 0) epi(row, acc);
}

// 3x1 blocks: B^T (interior P2 node rows, P1 columns), for K right-hand sides
// (x: K components, y: 3K component-major components)
template <int G, int K, class T, class Epi>
__global__ void __launch_bounds__(256) k_bt(int rows, const int* __restrict__ rp, const int* __restrict__ col,
                                            const T* __restrict__ v, long long nnz, const T* __restrict__ x, size_t xs,
                                            Epi epi) {
  dep_wait();
  constexpr int U = Batch<G>::U;
  int gt = blockIdx.x * blockDim.x + threadIdx.x;
  int row = gt / G, lane = gt & (G - 1);
  T acc[3 * K];
#pragma unroll
  for (int q = 0; q < 3 * K; ++q) acc[q] = T(0);
  if (row < rows) {
    const int e = rp[row + 1];
    for (int k = rp[row] + lane; k < e; k += U * G) {
      int c[U];
      T a[U][3];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int kk = k + u * G;
        const bool ok = kk < e;
        const int ks = ok ? kk : e - 1;  // in-bounds re-read, zero contribution
        c[u] = col[ks];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const T av = v[(size_t)j * nnz + ks];
          a[u][j] = ok ? av : T(0);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int q = 0; q < K; ++q) {
          const T xv = x[(size_t)q * xs + c[u]];
#pragma unroll
          for (int j = 0; j < 3; ++j) acc[3 * q + j] += a[u][j] * xv;
        }
    }
  }
  group_reduce<G, T, 3 * K>(acc);
  if (row < rows && lane == 0) epi(row, acc);
}

static_assert(kStencilVec == 4, "the stencil kernel loads four entries' weights per vector");
template <class T> struct Vec4;
template <> struct Vec4<float> { using type = float4; };
template <> struct Vec4<double> { using type = double4; };
__device__ __forceinline__ float4 ldcs_vec(const float4* p) { return __ldcs(p); }
__device__ __forceinline__ double4 ldcs_vec(const double4* p) {
  const double2* q = reinterpret_cast<const double2*>(p);
  const double2 a = __ldcs(q), b = __ldcs(q + 1);
  return make_double4(a.x, a.y, b.x, b.y);
}

// Stencil-structured product (StencilOp): one thread per row; a block holds
// rows of one class, so the entry loop, offsets and strides are uniform
// across the warp and consecutive lanes gather from nodes 2 apart.
// Fast path: if every y neighbour is inside the index space and every z
// neighbour is strictly inside (not on the first or last z plane), then for any
// x offset in [-2, 2] the neighbour index row + lin[e] lies in [0, size): the
// smallest reachable index is >= m - 2 and the largest <= m^3 - m^2 + 1 (m the
// points per axis). An x-neighbour outside the space may wrap into the
// adjacent line, but its stored weight is exactly 0. So rows need no test
// except near the y/z boundary, and no warp diverges at x-line ends.
#ifndef SK_ST_BLOCK
#define SK_ST_BLOCK 128  // threads per block of the stencil kernel
#endif
#ifndef SK_ST_UNROLL
#define SK_ST_UNROLL 2   // 4-entry groups unrolled (their loads in flight together)
#endif
constexpr int kStUnroll = SK_ST_UNROLL;
template <int NR, class TM, class T, class Epi>
__global__ void __launch_bounds__(SK_ST_BLOCK) k_stencil(const StArgs a, const TM* __restrict__ v, const T* __restrict__ x,
                                                 size_t xs, Epi epi) {
  dep_wait();
  int c, r;
  if (!st_locate(a, c, r)) return;
  int i, qx, qy, qz;
  st_coords(a, c, r, i, qx, qy, qz);
  if (i >= a.ext[c][0]) return;  // padding row
  const int row = st_index(a, qx, qy, qz);
  T acc[NR];
#pragma unroll
  for (int q = 0; q < NR; ++q) acc[q] = T(0);
  // kStencilVec consecutive entries' weights per vector load
  using V4 = typename Vec4<TM>::type;
  const V4* vr = reinterpret_cast<const V4*>(v + a.voff[c]) + r;
  const size_t rc = (size_t)a.prows[c];
  const int S4 = a.S[c] / kStencilVec, db = a.dbeg[c];
  // Entries whose neighbour lies outside the index space are stored as 0; their
  // linear index may fall on another node or, near the first and last planes,
  // outside the vector, so it is clamped into [0, xs): every row takes the same
  // branch-free loop and the zero weight cancels the clamped read.
  const int last = (int)xs - 1;
#pragma unroll kStUnroll
  for (int e4 = 0; e4 < S4; ++e4) {
    const V4 w4 = ldcs_vec(&vr[e4 * rc]);  // streamed once: evict first
    const TM wv[4] = {w4.x, w4.y, w4.z, w4.w};
    size_t cc[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) cc[j] = (size_t)min(max(row + a.lin[db + 4 * e4 + j], 0), last);
    if constexpr (Epi::il) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        T xv[NR];
        ldv<T, NR>(x + cc[j] * NR, xv);
        if constexpr (is_first<Epi>::value) {
          const T f = epi.gather_scale(cc[j]);
#pragma unroll
          for (int q = 0; q < NR; ++q) xv[q] *= f;
        }
#pragma unroll
        for (int q = 0; q < NR; ++q) acc[q] += (T)wv[j] * xv[q];
      }
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        // (fused first step: the gathered value times s0 D^-1 at its column,
        // rounded as the stored first iterate would be)
        T f = T(1);
        if constexpr (is_first<Epi>::value) f = epi.gather_scale(cc[j]);
#pragma unroll
        for (int q = 0; q < NR; ++q) {
          T xv = x[q * xs + cc[j]];
          if constexpr (is_first<Epi>::value) xv *= f;
          acc[q] += (T)wv[j] * xv;
        }
      }
    }
  }
  epi(row, acc);
}

// The same with the entry groups of a row spread over the W warps of a block of
// 32 rows (warp w takes groups w, w + W, ...) and the W partial sums added in
// shared memory: a thread per row leaves small levels latency-bound (one long
// chain of loads per row, or in FP64 of multiply-adds) and large ones idle in
// their last wave. Component-major rows end with a warp per component.
template <int NR, int W, class TM, class T, class Epi>
__global__ void __launch_bounds__(32 * W) k_stencil_w(const StArgs a, const TM* __restrict__ v,
                                                      const T* __restrict__ x, size_t xs, Epi epi) {
  dep_wait();
  __shared__ T sh[W][NR][32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int c = 0;
#pragma unroll 1
  while (c + 1 < a.ncls && (int)blockIdx.x >= a.bbeg[c + 1]) ++c;
  const int r = ((int)blockIdx.x - a.bbeg[c]) * 32 + lane;
  const bool live = r < a.rows[c];
  const int rr = live ? r : a.rows[c] - 1;
  const int line = (int)((rr * a.Mx[c]) >> 44), iz = (int)((line * a.My[c]) >> 44);  // FastDiv by the class's extents
  const int row = st_index(a, a.q0[c][0] + 2 * (rr - line * a.ext[c][0]), a.q0[c][1] + 2 * (line - iz * a.ext[c][1]),
                           a.q0[c][2] + 2 * iz);
  T acc[NR];
#pragma unroll
  for (int q = 0; q < NR; ++q) acc[q] = T(0);
  using V4 = typename Vec4<TM>::type;
  const V4* vr = reinterpret_cast<const V4*>(v + a.voff[c]) + rr;
  const size_t rc = (size_t)a.prows[c];
  const int S4 = a.S[c] / kStencilVec, db = a.dbeg[c], last = (int)xs - 1;
#pragma unroll 2
  for (int e4 = w; e4 < S4; e4 += W) {
    const V4 w4 = vr[e4 * rc];
    const TM wv[4] = {w4.x, w4.y, w4.z, w4.w};
    size_t cc[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) cc[j] = (size_t)min(max(row + a.lin[db + 4 * e4 + j], 0), last);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      T xv[NR];
      if constexpr (Epi::il) {
        ldv<T, NR>(x + cc[j] * NR, xv);
      } else {
#pragma unroll
        for (int q = 0; q < NR; ++q) xv[q] = x[q * xs + cc[j]];
      }
      if constexpr (is_first<Epi>::value) {
        const T f = epi.gather_scale(cc[j]);
#pragma unroll
        for (int q = 0; q < NR; ++q) xv[q] *= f;
      }
#pragma unroll
      for (int q = 0; q < NR; ++q) acc[q] += (T)wv[j] * xv[q];
    }
  }
#pragma unroll
  for (int q = 0; q < NR; ++q) sh[w][q][lane] = acc[q];
  __syncthreads();
  auto sum = [&](int q) {
    T s[W];
#pragma unroll
    for (int u = 0; u < W; ++u) s[u] = sh[u][q][lane];
#pragma unroll
    for (int o = W / 2; o; o >>= 1)
#pragma unroll
      for (int u = 0; u < o; ++u) s[u] += s[u + o];
    return s[0];
  };
  if constexpr (Epi::il) {
    if (w == 0 && live) {
#pragma unroll
      for (int q = 0; q < NR; ++q) acc[q] = sum(q);
      epi(row, acc);
    }
  } else {
    for (int q = w; q < NR; q += W) {
      const T s = sum(q);
      if (live) epi.comp(row, q, s);
    }
  }
}

// Warps per 32 rows (the lines and their measurements: internal.h)
template <class T> static inline int stencil_warps(long long rows, bool il) {
  const long long* lines = il ? kStencilSplitIL : (sizeof(T) == 8 ? kStencilSplit64 : kStencilSplit32);
  for (int k = 0; k < 3; ++k)
    if (rows < lines[k]) return 8 >> k;
  return 1;
}

template <int W, class T, class Epi>
static void launch_stencil_w(const Exec& ex, const StencilOp& so, const T* x, const Epi& epi, bool split, size_t xs) {
  const StArgs a = stencil_args(so, 32, 1, split);
  const int grid = a.bbeg[so.ncls];
  if (grid == 0) return;
  launch_dep(k_stencil_w<Epi::nr, W, T, T, Epi>, grid, 32 * W, 0, ex, a, so.template v<T>(), x, xs, epi);
}

template <class T, class Epi>
static void launch_stencil(const Exec& ex, const StencilOp& so, int nr, const T* x, const Epi& epi,
                           bool split = false) {
  size_t xs = 0;
  for (int c = 0; c < so.ncls; ++c) xs += so.rows[c];
  (void)nr;
  const int W = stencil_warps<T>((long long)xs, Epi::il);
  if (W == 8) return launch_stencil_w<8>(ex, so, x, epi, split, xs);
  if (W == 4) return launch_stencil_w<4>(ex, so, x, epi, split, xs);
  if (W == 2) return launch_stencil_w<2>(ex, so, x, epi, split, xs);
  const int bs = SK_ST_BLOCK;
  StArgs a = stencil_args(so, bs, kStencilRows, split);
  int grid = a.bbeg[so.ncls];
  if (grid == 0) return;
  launch_dep(k_stencil<Epi::nr, T, T, Epi>, grid, bs, 0, ex, a, so.template v<T>(), x, xs, epi);
  SK_CHECK_LAUNCH();
}

template <class T> static inline bool use_stencil(const Csr& m, bool il) {
  return m.st != nullptr && m.st->template v<T>() != nullptr && (il || m.rows >= m.st_min_single);
}

// algorithmic bytes: the matrix's stored entries (not the zero padding), x
// gathered once, the output and the epilogue's other vectors once
static double stencil_bytes(const StencilOp& so, int esz, int nr, int streams) {
  long long rows = 0;
  for (int c = 0; c < so.ncls; ++c) rows += so.rows[c];
  return (double)so.total_real * esz + (double)esz * rows * nr * (1 + streams);
}

// ---------------------------------------------------------------------------
// dispatch
// ---------------------------------------------------------------------------
enum Shape { SH_CSR = 0, SH_BSR3 = 2, SH_B = 3, SH_BT = 4 };  // CSR: right-hand sides from the epilogue

template <int G, class T, class Epi>
static void launch_g(const Exec& ex, const Csr& m, Shape sh, const T* x, const Epi& epi) {
  const int bs = 256;
  int grid = cdiv((long long)m.rows * G, bs);
  if (grid == 0) return;
  switch (sh) {
    case SH_CSR:
      launch_dep(k_csr<G, Epi::nr, T, T, Epi>, grid, bs, 0, ex, m.rows, m.rowptr, m.col, m.template v<T>(), x, m.cols, epi);
      break;
    case SH_BSR3:
      if constexpr (Epi::nr == 3)
        launch_dep(k_bsr3<G, T, Epi>, grid, bs, 0, ex, m.rows, m.rowptr, m.col, m.template v<T>(), m.nnz, x, m.cols, epi);
      break;
    case SH_B:
      if constexpr (Epi::nr == 1 || Epi::nr == 4)
        launch_dep(k_b<G, Epi::nr, T, Epi>, grid, bs, 0, ex, m.rows, m.rowptr, m.col, m.template v<T>(), m.nnz, x, m.cols,
                                                       epi);
      break;
    case SH_BT:
      if constexpr (Epi::nr == 3 || Epi::nr == 12)
        launch_dep(k_bt<G, Epi::nr / 3, T, Epi>, grid, bs, 0, ex, m.rows, m.rowptr, m.col, m.template v<T>(), m.nnz, x,
                                                            m.cols, epi);
      break;
  }
  SK_CHECK_LAUNCH();
}

template <class T, class Epi>
static void launch(const Exec& ex, const Csr& m, Shape sh, const T* x, const Epi& epi, int g) {
  SK_REQUIRE(m.template v<T>() != nullptr, STOKES_ERR_ARG, "matrix values missing for this precision");
  switch (g) {
    case 1: launch_g<1>(ex, m, sh, x, epi); break;
    case 2: launch_g<2>(ex, m, sh, x, epi); break;
    case 4: launch_g<4>(ex, m, sh, x, epi); break;
    case 8: launch_g<8>(ex, m, sh, x, epi); break;
    case 16: launch_g<16>(ex, m, sh, x, epi); break;
    default: launch_g<32>(ex, m, sh, x, epi); break;
  }
}

// bytes: matrix once + x once (cols*NR) + y once (rows*NR) (+ extra epilogue streams)
static double prod_bytes(const Csr& m, int esz, int nr_in, int nr_out, int extra_streams) {
  return m.bytes(esz) + (double)esz * ((double)m.cols * nr_in + (double)m.rows * nr_out * (1 + extra_streams));
}

// calls f(std::integral_constant<int, NR>) for the supported right-hand-side
// counts: 1 and 3 (one pressure or velocity vector), 4 and 12 (four of them)
template <class F> static void with_nr(int nr, F&& f) {
  switch (nr) {
    case 1: f(std::integral_constant<int, 1>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 12: f(std::integral_constant<int, 12>()); break;
    default: throw Error(STOKES_ERR_ARG, "sparse product: unsupported number of right-hand sides");
  }
}

// il: node-interleaved vectors (NR = 4 or 12 only), else component-major
template <int NR> static constexpr bool il_ok() { return NR % 4 == 0; }
static void require_il(int nr, bool il) {
  SK_REQUIRE(!il || nr % 4 == 0, STOKES_ERR_ARG, "interleaved vectors need 4 or 12 components");
}
template <class T, class E>
static void run_scalar(const Exec& ex, const Csr& m, bool st, const T* x, const E& e, bool split = false) {
  SK_REQUIRE(!split || (st && m.st->p2), STOKES_ERR_ARG, "parity-split products need P2 stencil storage");
  if (st) launch_stencil(ex, *m.st, E::nr, x, e, split);
  else launch(ex, m, SH_CSR, x, e, m.group);
}
template <class T> void spmv_store(const Exec& ex, const Csr& m, int nr, const T* x, T* y, int kind, int layout) {
  const bool il = layout & kLayoutIL, split = layout & kLayoutSplit;
  require_il(nr, il);
  const bool st = use_stencil<T>(m, il);
  ProfScope ps(ex, kind, st ? stencil_bytes(*m.st, sizeof(T), nr, 0) : prod_bytes(m, sizeof(T), nr, nr, 0));
  with_nr(nr, [&](auto NRc) {
    constexpr int NR = decltype(NRc)::value;
    if constexpr (il_ok<NR>()) {
      if (il) return run_scalar(ex, m, st, x, EpiStoreIL<T, NR>{y}, split);
    }
    run_scalar(ex, m, st, x, EpiStore<T, NR>{y, (size_t)m.rows}, split);
  });
}
template <class T> void spmv_add(const Exec& ex, const Csr& m, int nr, const T* x, T* y, int kind, int layout) {
  const bool il = layout & kLayoutIL, split = layout & kLayoutSplit;
  require_il(nr, il);
  const bool st = use_stencil<T>(m, il);
  ProfScope ps(ex, kind, st ? stencil_bytes(*m.st, sizeof(T), nr, 1) : prod_bytes(m, sizeof(T), nr, nr, 1));
  with_nr(nr, [&](auto NRc) {
    constexpr int NR = decltype(NRc)::value;
    if constexpr (il_ok<NR>()) {
      if (il) return run_scalar(ex, m, st, x, EpiAddIL<T, NR>{y}, split);
    }
    run_scalar(ex, m, st, x, EpiAdd<T, NR>{y, (size_t)m.rows}, split);
  });
}
template <class T>
void spmv_resid(const Exec& ex, const Csr& m, int nr, const T* b, const T* x, T* y, int kind, int layout) {
  const bool il = layout & kLayoutIL, split = layout & kLayoutSplit;
  require_il(nr, il);
  const bool st = use_stencil<T>(m, il);
  ProfScope ps(ex, kind, st ? stencil_bytes(*m.st, sizeof(T), nr, 1) : prod_bytes(m, sizeof(T), nr, nr, 1));
  with_nr(nr, [&](auto NRc) {
    constexpr int NR = decltype(NRc)::value;
    if constexpr (il_ok<NR>()) {
      if (il) return run_scalar(ex, m, st, x, EpiResidIL<T, NR>{b, y}, split);
    }
    run_scalar(ex, m, st, x, EpiResid<T, NR>{b, y, (size_t)m.rows}, split);
  });
}
template <class T> void spmv_cheb(const Exec& ex, const Csr& m, int nr, const T* b, const T* xin, T* d, T* xout,
                                  const T* dinv, double c1, double c2, int kind, int layout) {
  const bool il = layout & kLayoutIL, split = layout & kLayoutSplit;
  require_il(nr, il);
  const bool st = use_stencil<T>(m, il);
  // streams: b, x_in (own row), d read, d write, x_out write, dinv
  ProfScope ps(ex, kind,
               (st ? stencil_bytes(*m.st, sizeof(T), nr, 4) : prod_bytes(m, sizeof(T), nr, nr, 4)) +
                   (double)sizeof(T) * m.rows);
  with_nr(nr, [&](auto NRc) {
    constexpr int NR = decltype(NRc)::value;
    if constexpr (il_ok<NR>()) {
      if (il) return run_scalar(ex, m, st, xin, EpiChebIL<T, NR>{b, xin, d, xout, dinv, (T)c1, (T)c2}, split);
    }
    run_scalar(ex, m, st, xin, EpiCheb<T, NR>{b, xin, d, xout, dinv, (T)c1, (T)c2, (size_t)m.rows}, split);
  });
}
template <class T> void spmv_cheb_first(const Exec& ex, const Csr& m, int nr, const T* b, T* d, T* xout,
                                        const T* dinv, double s0, double c1, double c2, int kind, int layout) {
  const bool il = layout & kLayoutIL, split = layout & kLayoutSplit;
  require_il(nr, il);
  const bool st = use_stencil<T>(m, il);
  // streams: b gathered, d and x_out written, D^-1 gathered
  ProfScope ps(ex, kind,
               (st ? stencil_bytes(*m.st, sizeof(T), nr, 2) : prod_bytes(m, sizeof(T), nr, nr, 2)) +
                   (double)sizeof(T) * m.rows);
  with_nr(nr, [&](auto NRc) {
    constexpr int NR = decltype(NRc)::value;
    if constexpr (il_ok<NR>()) {
      if (il) return run_scalar(ex, m, st, b, EpiChebFirstIL<T, NR>{b, d, xout, dinv, (T)s0, (T)c1, (T)c2}, split);
    }
    run_scalar(ex, m, st, b, EpiChebFirst<T, NR>{b, d, xout, dinv, (T)s0, (T)c1, (T)c2, (size_t)m.rows}, split);
  });
}
template <class T> bool stencil_in_use(const Csr& m, bool il) { return use_stencil<T>(m, il); }

template <class T>
void restrict_split(const Exec& ex, const Csr& R, int nr, const T* x, T* y, bool il, const SplitMap& sm) {
  require_il(nr, il);
  ProfScope ps(ex, STOKES_KERNEL_TRANSFER, prod_bytes(R, sizeof(T), nr, nr, 0));
  with_nr(nr, [&](auto NRc) {
    constexpr int NR = decltype(NRc)::value;
    if constexpr (il_ok<NR>()) {
      if (il) return launch(ex, R, SH_CSR, x, WithColMap<EpiStoreIL<T, NR>>{{y}, sm}, R.group);
    }
    launch(ex, R, SH_CSR, x, WithColMap<EpiStore<T, NR>>{{y, (size_t)R.rows}, sm}, R.group);
  });
}
void prolong_add_split(const Exec& ex, const Csr& P, int nr, const double* x, double* y, bool il, const SplitMap& sm) {
  using T = double;
  require_il(nr, il);
  ProfScope ps(ex, STOKES_KERNEL_TRANSFER, prod_bytes(P, sizeof(T), nr, nr, 1));
  with_nr(nr, [&](auto NRc) {
    constexpr int NR = decltype(NRc)::value;
    if constexpr (il_ok<NR>()) {
      if (il) return launch(ex, P, SH_CSR, x, WithRowMap<EpiAddIL<T, NR>>{{y}, sm}, P.group);
    }
    launch(ex, P, SH_CSR, x, WithRowMap<EpiAdd<T, NR>>{{y, (size_t)P.rows}, sm}, P.group);
  });
}
template <class T> void bsr3_cheb(const Exec& ex, const Csr& m, const T* b, const T* xin, T* d, T* xout,
                                  const T* dinv, double c1, double c2, int kind) {
  // streams as in the scalar step, over 3 components and a 3-component diagonal
  ProfScope ps(ex, kind, prod_bytes(m, sizeof(T), 3, 3, 4) + 3.0 * sizeof(T) * m.rows);
  launch(ex, m, SH_BSR3, xin, EpiCheb3<T>{b, xin, d, xout, dinv, (T)c1, (T)c2, (size_t)m.rows}, m.group);
}
// FP32 products of A run element by element (element.cu) wherever the context
// has the geometry (mixed precision, formats 0 and 2): faster than the stored
// blocks on every mesh measured, 8^3 to 96^3 (figures there)
template <class T> static inline bool use_element(const Csr& m) {
  return std::is_same<T, float>::value && m.el && m.sym_products;
}
// geometry once, x gathered once, y and `streams` further vectors once
static double element_bytes(const ElementOp& e, int rows, int k, int streams) {
  return 4.0 * (6.0 * kElWords * e.n * e.n * e.n + 3.0 * rows * k * (2 + streams));
}
template <class T> void bsr3_apply(const Exec& ex, const Csr& m, const T* x, T* y, const T* b, int kind) {
  if constexpr (std::is_same<T, float>::value) {
    if (use_element<T>(m)) {
      ProfScope ps(ex, kind, element_bytes(*m.el, m.rows, 1, b ? 1 : 0));
      element_strain(ex, *m.el, 1, x, y, b, nullptr, nullptr);
      return;
    }
  }
  if constexpr (std::is_same<T, double>::value) {
    if (m.sym && m.sym_products) {
      ProfScope ps(ex, kind, sym3_bytes(*m.sym, sizeof(T), m.rows, b ? 1 : 0));
      sym3_launch(ex, m, x, y, b, nullptr, nullptr);
      return;
    }
  }
  ProfScope ps(ex, kind, prod_bytes(m, sizeof(T), 3, 3, b ? 1 : 0));
  if (b) launch(ex, m, SH_BSR3, x, EpiResid<T, 3>{b, y, (size_t)m.rows}, m.group);
  else launch(ex, m, SH_BSR3, x, EpiStore<T, 3>{y, (size_t)m.rows}, m.group);
}
template <class T>
void bsr3_apply_k(const Exec& ex, const Csr& m, int k, const T* x, T* y, const T* b, int kind) {
  if constexpr (std::is_same<T, float>::value) {
    if (use_element<T>(m)) {
      ProfScope ps(ex, kind, element_bytes(*m.el, m.rows, k, b ? 1 : 0));
      element_strain(ex, *m.el, k, x, y, b, nullptr, nullptr);
      return;
    }
  }
  if constexpr (std::is_same<T, double>::value) {
    if (k == 4 && m.sym && m.sym_products) {
      ProfScope ps(ex, kind, (double)m.sym->total * sizeof(T) + (double)sizeof(T) * 3.0 * m.rows * 4 * (b ? 2 : 1));
      sym3_launch4(ex, m, x, y, b);
      return;
    }
  }
  const size_t len = 3 * (size_t)m.rows;
  for (int i = 0; i < k; ++i) bsr3_apply<T>(ex, m, x + i * len, y + i * len, b ? b + i * len : nullptr, kind);
}
template <class T> bool bsr3_apply_dot(const Exec& ex, const Csr& m, const T* x, T* y, const DotScratch& ds,
                                       double* dot) {
  if constexpr (std::is_same<T, float>::value) {
    if (use_element<T>(m)) {
      ProfScope ps(ex, STOKES_KERNEL_SPMV_A, element_bytes(*m.el, m.rows, 1, 1));
      element_strain(ex, *m.el, 1, x, y, nullptr, &ds, dot);
      return true;
    }
  }
  if constexpr (std::is_same<T, double>::value) {
    if (m.sym && m.sym_products && ds.fused_partial && sym3_grid(*m.sym) <= ds.fused_cap) {
      // the product's bytes plus the own-row x read of the fused dot
      ProfScope ps(ex, STOKES_KERNEL_SPMV_A, sym3_bytes(*m.sym, sizeof(T), m.rows, 1));
      sym3_launch(ex, m, x, y, (const T*)nullptr, &ds, dot);
      return true;
    }
  }
  if (m.template v<T>() && ds.fused_partial && bsr3_dot_grid(m) <= ds.fused_cap) {
    ProfScope ps(ex, STOKES_KERNEL_SPMV_A, prod_bytes(m, sizeof(T), 3, 3, 1));
    switch (m.group) {
      case 1: launch_bsr3_dot<1, T>(ex, m, x, y, ds, dot); break;
      case 2: launch_bsr3_dot<2, T>(ex, m, x, y, ds, dot); break;
      case 4: launch_bsr3_dot<4, T>(ex, m, x, y, ds, dot); break;
      case 8: launch_bsr3_dot<8, T>(ex, m, x, y, ds, dot); break;
      case 16: launch_bsr3_dot<16, T>(ex, m, x, y, ds, dot); break;
      default: launch_bsr3_dot<32, T>(ex, m, x, y, ds, dot); break;
    }
    return true;
  }
  bsr3_apply<T>(ex, m, x, y, (const T*)nullptr);
  const T* xs[1] = {x};
  const T* ys[1] = {y};
  dots<T>(ex, ds, 1, xs, ys, (size_t)m.rows * 3, dot, kDotFast);
  return false;
}

template <class T>
void bsr3_apply_dot_k(const Exec& ex, const Csr& m, int k, const T* x, T* y, const DotScratch& ds, double* dot) {
  if constexpr (std::is_same<T, float>::value) {
    if (use_element<T>(m)) {
      ProfScope ps(ex, STOKES_KERNEL_SPMV_A, element_bytes(*m.el, m.rows, k, 1));
      element_strain(ex, *m.el, k, x, y, nullptr, &ds, dot);
      return;
    }
  }
  const size_t len = 3 * (size_t)m.rows;
  for (int i = 0; i < k; ++i) bsr3_apply_dot<T>(ex, m, x + i * len, y + i * len, ds, dot + i);
}

template <class T> void b_apply(const Exec& ex, const Csr& m, const T* x, T* y, const T* b, double alpha, int k) {
  SK_REQUIRE(k == 1 || k == 4, STOKES_ERR_ARG, "B product: 1 or 4 right-hand sides");
  if (m.div) {  // the stored values once (its zero blocks not counted)
    ProfScope ps(ex, STOKES_KERNEL_B, sizeof(T) * (3.0 * m.nnz + k * (3.0 * m.cols + m.rows * (b ? 2.0 : 1.0))));
    div_apply<T>(ex, *m.div, k, x, y, b, alpha);
    return;
  }
  ProfScope ps(ex, STOKES_KERNEL_B, m.bytes(sizeof(T)) + sizeof(T) * k * (3.0 * m.cols + m.rows * (b ? 2.0 : 1.0)));
  if (k == 4) launch(ex, m, SH_B, x, EpiAxpy<T, 4>{b, nullptr, y, (T)alpha, (size_t)m.rows}, m.group4 ? m.group4 : m.group);
  else launch(ex, m, SH_B, x, EpiAxpy<T, 1>{b, nullptr, y, (T)alpha, (size_t)m.rows}, m.group);
}
template <class T> void bt_apply(const Exec& ex, const Csr& m, const T* x, T* y, const T* scale, const T* b,
                                 double alpha, int k) {
  SK_REQUIRE(k == 1 || k == 4, STOKES_ERR_ARG, "B^T product: 1 or 4 right-hand sides");
  if (m.div) {
    ProfScope ps(ex, STOKES_KERNEL_BT, sizeof(T) * (3.0 * m.nnz + k * (1.0 * m.cols + 3.0 * m.rows * (b ? 2.0 : 1.0)) +
                                                    (scale ? m.rows : 0)));
    divt_apply<T>(ex, *m.div, k, x, y, scale, b, alpha);
    return;
  }
  ProfScope ps(ex, STOKES_KERNEL_BT,
               m.bytes(sizeof(T)) +
                   sizeof(T) * (k * (1.0 * m.cols + 3.0 * m.rows * (b ? 2.0 : 1.0)) + (scale ? m.rows : 0)));
  if (k == 4) launch(ex, m, SH_BT, x, EpiAxpy<T, 12>{b, scale, y, (T)alpha, (size_t)m.rows}, m.group4 ? m.group4 : m.group);
  else launch(ex, m, SH_BT, x, EpiAxpy<T, 3>{b, scale, y, (T)alpha, (size_t)m.rows}, m.group);
}

// coarse dense inverse applied to NR right-hand sides: one warp per row
template <int NR, class T, bool IL = false>
__global__ void k_dense(const T* __restrict__ M, int m, const T* __restrict__ b, T* __restrict__ y) {
  dep_wait();
  // component-major right-hand sides: component r of row j at r * m + j
  // (IL: node-interleaved, at j * NR + r)
  int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  int lane = threadIdx.x & 31;
  if (row >= m) return;
  T acc[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) acc[r] = T(0);
  for (int j = lane; j < m; j += 32) {
    T a = M[(size_t)row * m + j];
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r] += a * b[IL ? (size_t)j * NR + r : (size_t)r * m + j];
  }
#pragma unroll
  for (int o = 16; o; o >>= 1)
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
  if (lane == 0)
#pragma unroll
    for (int r = 0; r < NR; ++r) y[IL ? (size_t)row * NR + r : (size_t)r * m + row] = acc[r];
}

template <class T> void dense_apply(const Exec& ex, const T* Minv, int m, int nr, const T* b, T* y, bool il) {
  ProfScope ps(ex, STOKES_KERNEL_OTHER, (double)sizeof(T) * ((double)m * m + 2.0 * m * nr));
  int grid = cdiv(m, 8);
  with_nr(nr, [&](auto NRc) {
    constexpr int NR = decltype(NRc)::value;
    if (il) launch_dep(k_dense<NR, T, true>, grid, 256, 0, ex, Minv, m, b, y);
    else launch_dep(k_dense<NR, T, false>, grid, 256, 0, ex, Minv, m, b, y);
  });
  SK_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------
// autotuner: time each group width on this matrix, keep the fastest. Results
// are cached per (device, kernel shape, precision, matrix size) in a text file
// (STOKES_TUNE_CACHE, else _build/tune_cache.txt next to the library), so a
// later process - for example the same benchmark under a profiler, whose
// serialised launches would distort the timings - reuses the decision.
// ---------------------------------------------------------------------------
constexpr int kTuneVersion = 2;  // bump when the kernels change

static std::mutex g_tune_mutex;
static std::map<std::string, int>* g_tune = nullptr;

static std::string tune_cache_path() {
  const char* env = std::getenv("STOKES_TUNE_CACHE");
  if (env && *env) return env;
  Dl_info info;
  if (dladdr((void*)&tune_cache_path, &info) && info.dli_fname) {
    std::string f = info.dli_fname;
    size_t slash = f.rfind('/');
    if (slash != std::string::npos) return f.substr(0, slash) + "/_build/tune_cache.txt";
  }
  return "";
}

static void tune_load() {
  if (g_tune) return;
  g_tune = new std::map<std::string, int>();
  std::string path = tune_cache_path();
  if (path.empty()) return;
  FILE* fh = std::fopen(path.c_str(), "r");
  if (!fh) return;
  char key[512];
  int g;
  while (std::fscanf(fh, "%511s %d", key, &g) == 2) (*g_tune)[key] = g;
  std::fclose(fh);
}

static void tune_store(const std::string& key, int g) {
  (*g_tune)[key] = g;
  std::string path = tune_cache_path();
  if (path.empty()) return;
  FILE* fh = std::fopen(path.c_str(), "a");
  if (!fh) return;  // read-only location: keep the in-process decision only
  std::fprintf(fh, "%s %d\n", key.c_str(), g);
  std::fclose(fh);
}

void autotune_group(const Exec& ex, Csr& m, int nr, int kind, int k) {
  if (m.rows == 0) return;
  Shape sh = kind == 1 ? SH_BSR3 : kind == 2 ? SH_B : kind == 3 ? SH_BT : SH_CSR;
  SK_REQUIRE(k == 1 || ((sh == SH_B || sh == SH_BT) && k == 4), STOKES_ERR_ARG,
             "autotuner: four right-hand sides for B and B^T only");
  int xin = k * ((sh == SH_BSR3 || sh == SH_B) ? 3 : (sh == SH_BT ? 1 : nr));
  int yout = k * ((sh == SH_BSR3 || sh == SH_BT) ? 3 : (sh == SH_B ? 1 : nr));
  int& slot = k > 1 ? m.group4 : m.group;
  bool f32 = m.v64 == nullptr;
  size_t esz = f32 ? 4 : 8;
  int dev = 0;
  SK_CUDA(cudaGetDevice(&dev));
  cudaDeviceProp prop;
  SK_CUDA(cudaGetDeviceProperties(&prop, dev));
  std::string devname = prop.name;
  for (char& ch : devname)
    if (ch == ' ') ch = '_';
  char key[512];
  std::snprintf(key, sizeof(key), "v%d|%s|sh%d|f%d|r%d|c%d|z%lld%s", kTuneVersion, devname.c_str(), (int)sh,
                f32 ? 32 : 64, m.rows, m.cols, (long long)m.nnz, k > 1 ? "|k4" : "");
  {
    std::lock_guard<std::mutex> lock(g_tune_mutex);
    tune_load();
    auto it = g_tune->find(key);
    if (it != g_tune->end()) {
      slot = it->second;
      return;
    }
  }
  void *x = nullptr, *y = nullptr;
  SK_CUDA(cudaMalloc(&x, esz * (size_t)m.cols * xin));
  SK_CUDA(cudaMalloc(&y, esz * (size_t)m.rows * yout));
  SK_CUDA(cudaMemsetAsync(x, 0, esz * (size_t)m.cols * xin, ex.s));
  cudaEvent_t e0, e1;
  SK_CUDA(cudaEventCreate(&e0));
  SK_CUDA(cudaEventCreate(&e1));
  Exec plain{ex.s, nullptr};
  plain.dep = false;  // time launches on their own, not overlapped with the next
  float best = FLT_MAX;
  int bestg = slot ? slot : m.group;
  const int gs[5] = {2, 4, 8, 16, 32};
  for (int gi = 0; gi < 5; ++gi) {
    int g = gs[gi];
    auto run = [&]() {
      with_nr(yout, [&](auto NRc) {
        constexpr int NR = decltype(NRc)::value;
        if (f32) launch(plain, m, sh, (const float*)x, EpiStore<float, NR>{(float*)y, (size_t)m.rows}, g);
        else launch(plain, m, sh, (const double*)x, EpiStore<double, NR>{(double*)y, (size_t)m.rows}, g);
      });
    };
    run();
    float gbest = FLT_MAX;
    for (int trial = 0; trial < 3; ++trial) {
      SK_CUDA(cudaEventRecord(e0, ex.s));
      for (int rep = 0; rep < 3; ++rep) run();
      SK_CUDA(cudaEventRecord(e1, ex.s));
      SK_CUDA(cudaEventSynchronize(e1));
      float ms = 0;
      SK_CUDA(cudaEventElapsedTime(&ms, e0, e1));
      gbest = std::min(gbest, ms);
    }
    if (gbest < best) best = gbest, bestg = g;
  }
  slot = bestg;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(x);
  cudaFree(y);
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  tune_store(key, bestg);
}

#define SK_INST(T)                                                                                        \
  template void spmv_store<T>(const Exec&, const Csr&, int, const T*, T*, int, int);                          \
  template void spmv_add<T>(const Exec&, const Csr&, int, const T*, T*, int, int);                            \
  template void spmv_resid<T>(const Exec&, const Csr&, int, const T*, const T*, T*, int, int);                \
  template void spmv_cheb<T>(const Exec&, const Csr&, int, const T*, const T*, T*, T*, const T*, double, \
                             double, int, int);                                                         \
  template void spmv_cheb_first<T>(const Exec&, const Csr&, int, const T*, T*, T*, const T*, double,      \
                                   double, double, int, int);                                          \
  template bool stencil_in_use<T>(const Csr&, bool);                                                     \
  template void restrict_split<T>(const Exec&, const Csr&, int, const T*, T*, bool, const SplitMap&);   \
  template void bsr3_apply<T>(const Exec&, const Csr&, const T*, T*, const T*, int);                          \
  template void bsr3_cheb<T>(const Exec&, const Csr&, const T*, const T*, T*, T*, const T*, double, double, int); \
  template void b_apply<T>(const Exec&, const Csr&, const T*, T*, const T*, double, int);                \
  template void bt_apply<T>(const Exec&, const Csr&, const T*, T*, const T*, const T*, double, int);     \
  template void dense_apply<T>(const Exec&, const T*, int, int, const T*, T*, bool);                    \
  template void bsr3_apply_k<T>(const Exec&, const Csr&, int, const T*, T*, const T*, int);            \
  template bool bsr3_apply_dot<T>(const Exec&, const Csr&, const T*, T*, const DotScratch&, double*);   \
  template void bsr3_apply_dot_k<T>(const Exec&, const Csr&, int, const T*, T*, const DotScratch&, double*);
SK_INST(float)
SK_INST(double)

}  // namespace sk
