// Products with the strain-form velocity operator A in symmetric stencil
// storage (Sym3Op): each row reads its diagonal and "upper" 3x3 blocks from its
// own storage and the transposes of its "lower" blocks from the neighbours'
// storage, so the stored values are half of the BSR3 values and carry no
// column indices.
//
// Launch order: blocks walk the half-grid z-planes in order and, within a
// plane, the four classes that have rows there. A lower block of row i
// (neighbour j at most one cube layer below i) was read directly by row j a
// few planes earlier, i.e. within the last few tens of MB of traffic, so the
// second read is served from L2 and each value crosses HBM about once.
#include <algorithm>
#include <cstdio>
#include <cstring>

#include "internal.h"

namespace sk {

struct Sym3Args {
  int m, hiq;                  // points per axis (2n-1); highest interior half-grid coordinate
  int bo, be;                  // blocks of an odd / even half-grid z-plane (all its classes)
  int nb[8];                   // blocks per (class, plane)
  int ext[8][3], q0[8][3], pext[8], prows[8], ubeg[9], lbeg[9];
  long long voff[8];
  signed char ud[kMaxSym][3];
  int ulin[kMaxSym];
  signed char ld[kMaxSym][3];
  int llin[kMaxSym];
  int lcls[kMaxSym];
  long long lbase[kMaxSym];
  signed char ldel[kMaxSym][3];
};

constexpr int kSymRows = 32;  // rows per block

static Sym3Args sym3_args(const Sym3Op& so) {
  Sym3Args a;
  std::memset(&a, 0, sizeof(a));
  a.m = 2 * so.n - 1;
  a.hiq = 2 * so.n - 1;
  for (int c = 0; c < 8; ++c) {
    for (int k = 0; k < 3; ++k) a.ext[c][k] = so.ext[c][k], a.q0[c][k] = so.q0[c][k];
    a.pext[c] = so.pext[c];
    a.prows[c] = so.prows[c];
    a.voff[c] = so.voff[c];
    a.nb[c] = cdiv((long long)so.pext[c] * so.ext[c][1], kSymRows);
  }
  for (int c = 0; c < 9; ++c) a.ubeg[c] = so.ubeg[c], a.lbeg[c] = so.lbeg[c];
  // classes with an odd z coordinate (bit 2 set) have rows on odd planes
  a.bo = a.nb[4] + a.nb[5] + a.nb[6] + a.nb[7];
  a.be = a.nb[0] + a.nb[1] + a.nb[2] + a.nb[3];
  for (int e = 0; e < so.ubeg[8]; ++e) {
    for (int k = 0; k < 3; ++k) a.ud[e][k] = so.ud[e][k];
    a.ulin[e] = so.ulin[e];
  }
  for (int e = 0; e < so.lbeg[8]; ++e) {
    for (int k = 0; k < 3; ++k) a.ld[e][k] = so.ld[e][k], a.ldel[e][k] = so.ldel[e][k];
    a.llin[e] = so.llin[e];
    a.lcls[e] = so.lcls[e];
    a.lbase[e] = so.lbase[e];
  }
  return a;
}

// n odd planes (qz = 1, 3, ..., 2n-1) and n-1 even planes (qz = 2, ..., 2n-2),
// interleaved: odd plane k, even plane k, odd plane k+1, ...
static int sym3_blocks(const Sym3Op& so, const Sym3Args& a) { return so.n * a.bo + (so.n - 1) * a.be; }
int sym3_grid(const Sym3Op& so) { return sym3_blocks(so, sym3_args(so)); }

struct SymRow {
  int c, ix, iy, iz, pr, row, qx, qy, qz;
  bool valid;
};

// row `slot` of virtual block vb, `rows` rows per block
__device__ __forceinline__ SymRow sym3_locate(const Sym3Args& a, int vb, int rows, int slot) {
  SymRow r;
  const int pair = vb / (a.bo + a.be);
  int rem = vb - pair * (a.bo + a.be);
  const bool odd = rem < a.bo;
  if (!odd) rem -= a.bo;
  int c = odd ? 4 : 0;
#pragma unroll 1
  for (int k = 0; k < 3 && rem >= a.nb[c]; ++k) rem -= a.nb[c++];
  r.c = c;
  r.iz = pair;  // odd planes: qz = 1 + 2 pair; even planes: qz = 2 + 2 pair
  const int plane = a.pext[c] * a.ext[c][1];
  const int t = rem * rows + slot;
  r.valid = t < plane;
  const int tt = r.valid ? t : 0;
  r.ix = tt % a.pext[c];
  r.iy = tt / a.pext[c];
  r.pr = r.iz * plane + tt;
  r.qx = a.q0[c][0] + 2 * r.ix;
  r.qy = a.q0[c][1] + 2 * r.iy;
  r.qz = a.q0[c][2] + 2 * r.iz;
  r.row = (r.qx - 1) + a.m * ((r.qy - 1) + a.m * (r.qz - 1));
  return r;
}

__device__ __forceinline__ bool sym3_inside(const Sym3Args& a, int x, int y, int z) {
  return x >= 1 && x <= a.hiq && y >= 1 && y <= a.hiq && z >= 1 && z <= a.hiq;
}

// Batched loads (as in the CSR kernels): a thread first issues the value loads of
// U entries (entries lane, lane + G, ..., lane + (U-1) G of its row, lane the
// thread's warp in the block), then their x gathers, then the FMAs, so that U
// block loads per thread are in flight per HBM round trip. Entries past the end
// re-read a valid entry and weigh 0.
// this thread's share of acc[3k + r] = sum over the row's blocks of
// A(i, j)_{r q} x_k,j[q] for K right-hand sides (x: 3K component-major
// components), U entries' loads in flight; each block is read once
// for all K
template <int G, int U, int K, class T>
__device__ __forceinline__ void sym3_row(const Sym3Args& a, const SymRow& R, int lane, const T* __restrict__ v,
                                         const T* __restrict__ x, size_t xs, T* acc) {
  const int c = R.c;
  const int last = (int)xs - 1;
  const size_t rc = (size_t)a.prows[c];
  const T* vr = v + a.voff[c] + R.pr;
  const int u0 = a.ubeg[c], nu = a.ubeg[c + 1] - u0;
  for (int e0 = lane; e0 < nu; e0 += U * G) {
    T w[U][9];
    int cc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * G;
      const bool ok = e < nu;
      const int es = ok ? e : nu - 1;
      cc[u] = min(max(R.row + a.ulin[u0 + es], 0), last);
      const T* vb = vr + (size_t)9 * es * rc;
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const T t = vb[k * rc];
        w[u][k] = ok ? t : T(0);
      }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const T* xk = x + (size_t)3 * k * xs;
      T xv[U][3];
#pragma unroll
      for (int u = 0; u < U; ++u) xv[u][0] = xk[cc[u]], xv[u][1] = xk[xs + cc[u]], xv[u][2] = xk[2 * xs + cc[u]];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int r = 0; r < 3; ++r)
          acc[3 * k + r] += w[u][3 * r] * xv[u][0] + w[u][3 * r + 1] * xv[u][1] + w[u][3 * r + 2] * xv[u][2];
    }
  }
  const int l0 = a.lbeg[c], nl = a.lbeg[c + 1] - l0;
  for (int e0 = lane; e0 < nl; e0 += U * G) {
    T w[U][9];
    int cc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * G;
      const int L = l0 + (e < nl ? e : nl - 1);
      const bool in = e < nl && sym3_inside(a, R.qx + a.ld[L][0], R.qy + a.ld[L][1], R.qz + a.ld[L][2]);
      const int cs = a.lcls[L];
      const int jx = R.ix + a.ldel[L][0], jy = R.iy + a.ldel[L][1], jz = R.iz + a.ldel[L][2];
      const int rj = in ? jx + a.pext[cs] * (jy + a.ext[cs][1] * jz) : 0;
      const size_t rcs = (size_t)a.prows[cs];
      const T* vb = v + a.lbase[L] + rj;
      cc[u] = min(max(R.row + a.llin[L], 0), last);
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const T t = vb[k * rcs];
        w[u][k] = in ? t : T(0);
      }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const T* xk = x + (size_t)3 * k * xs;
      T xv[U][3];
#pragma unroll
      for (int u = 0; u < U; ++u) xv[u][0] = xk[cc[u]], xv[u][1] = xk[xs + cc[u]], xv[u][2] = xk[2 * xs + cc[u]];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int r = 0; r < 3; ++r)
          acc[3 * k + r] += w[u][r] * xv[u][0] + w[u][3 + r] * xv[u][1] + w[u][6 + r] * xv[u][2];
    }
  }
}

// y = A x (b == nullptr) or y = b - A x; with DOT, *dot = x . (A x) over all rows.
// A block takes 32 rows; its warp w the entries w, w + W, ... of each, the
// partial sums are added in shared memory and a warp per component finishes.
// Blocks walk the virtual blocks (plane order) with a grid stride; the dot
// variant runs one resident wave so that its grid sum takes one counter
// increment per resident block.
// K right-hand sides: x, b, y hold 3K component-major components (the dot
// variant is K = 1 only)
template <int W, int U, class T, bool DOT, int K = 1>
__global__ void __launch_bounds__(32 * W) k_sym3(const Sym3Args a, int nvb, const T* __restrict__ v,
                                                 const T* __restrict__ x, size_t xs, const T* __restrict__ b,
                                                 T* __restrict__ y, double* partial, unsigned* counter, double* dot) {
  dep_wait();
  static_assert(!DOT || K == 1, "fused dot: one right-hand side");
  __shared__ T sh[W][3 * K][32];
  const int w = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  double part = 0.0;
  for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
    const SymRow R = sym3_locate(a, vb, kSymRows, lane);
    T acc[3 * K];
#pragma unroll
    for (int r = 0; r < 3 * K; ++r) acc[r] = T(0);
    if (R.valid) sym3_row<W, U, K, T>(a, R, w, v, x, xs, acc);
#pragma unroll
    for (int r = 0; r < 3 * K; ++r) sh[w][r][lane] = acc[r];
    __syncthreads();
    for (int r = w; r < 3 * K; r += W) {
      T s[W];
#pragma unroll
      for (int u = 0; u < W; ++u) s[u] = sh[u][r][lane];
#pragma unroll
      for (int o = W / 2; o; o >>= 1)
#pragma unroll
        for (int u = 0; u < o; ++u) s[u] += s[u + o];
      if (R.valid) {
        const size_t i = r * xs + R.row;
        y[i] = b ? b[i] - s[0] : s[0];
        if (DOT) part += (double)(s[0] * x[i]);
      }
    }
    __syncthreads();
  }
  if (DOT) grid_sum(part, partial, counter, dot);
}

// y = b - A x in double-float arithmetic: A = vh + vl, x = xh + xl (FP32
// pairs); K right-hand sides (x, b, y: 3K component-major components), each
// stored block read once for all K
template <int W, int U, int K>
__global__ void __launch_bounds__(32 * W) k_sym3_df(const Sym3Args a, const float* __restrict__ vh,
                                                      const float* __restrict__ vl, const float* __restrict__ xh,
                                                      const float* __restrict__ xl, size_t xs,
                                                      const double* __restrict__ b, double* __restrict__ y) {
  dep_wait();
  constexpr int G = W;
  __shared__ DF sh[W][3 * K][32];
  const int lane = (int)threadIdx.x >> 5, slot = (int)threadIdx.x & 31;  // (lane: the warp, as in sym3_row)
  const SymRow R = sym3_locate(a, (int)blockIdx.x, kSymRows, slot);
  const int c = R.c;
  const int last = (int)xs - 1;
  DF acc[3 * K];
#pragma unroll
  for (int r = 0; r < 3 * K; ++r) acc[r] = DF{0.f, 0.f};
  if (R.valid) {
    const size_t rc = (size_t)a.prows[c];
    const int u0 = a.ubeg[c], nu = a.ubeg[c + 1] - u0;
    for (int e0 = lane; e0 < nu; e0 += U * G) {
      float wh[U][9], wl[U][9];
      int cc[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + u * G;
        const bool ok = e < nu;
        const int es = ok ? e : nu - 1;
        cc[u] = min(max(R.row + a.ulin[u0 + es], 0), last);
        const size_t base = a.voff[c] + (size_t)9 * es * rc + R.pr;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          const float h = vh[base + k * rc], l = vl[base + k * rc];
          wh[u][k] = ok ? h : 0.f;
          wl[u][k] = ok ? l : 0.f;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int k = 0; k < K; ++k) {
          float x_h[3], x_l[3];
#pragma unroll
          for (int q = 0; q < 3; ++q) x_h[q] = xh[(3 * k + q) * xs + cc[u]], x_l[q] = xl[(3 * k + q) * xs + cc[u]];
#pragma unroll
          for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int q = 0; q < 3; ++q)
              df_madd(acc[3 * k + r], wh[u][3 * r + q], wl[u][3 * r + q], x_h[q], x_l[q]);
        }
    }
    const int l0 = a.lbeg[c], nl = a.lbeg[c + 1] - l0;
    for (int e0 = lane; e0 < nl; e0 += U * G) {
      float wh[U][9], wl[U][9];
      int cc[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + u * G;
        const int L = l0 + (e < nl ? e : nl - 1);
        const bool in = e < nl && sym3_inside(a, R.qx + a.ld[L][0], R.qy + a.ld[L][1], R.qz + a.ld[L][2]);
        const int cs = a.lcls[L];
        const int jx = R.ix + a.ldel[L][0], jy = R.iy + a.ldel[L][1], jz = R.iz + a.ldel[L][2];
        const int rj = in ? jx + a.pext[cs] * (jy + a.ext[cs][1] * jz) : 0;
        const size_t rcs = (size_t)a.prows[cs];
        const size_t base = a.lbase[L] + rj;
        cc[u] = min(max(R.row + a.llin[L], 0), last);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          const float h = vh[base + k * rcs], l = vl[base + k * rcs];
          wh[u][k] = in ? h : 0.f;
          wl[u][k] = in ? l : 0.f;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int k = 0; k < K; ++k) {
          float x_h[3], x_l[3];
#pragma unroll
          for (int q = 0; q < 3; ++q) x_h[q] = xh[(3 * k + q) * xs + cc[u]], x_l[q] = xl[(3 * k + q) * xs + cc[u]];
#pragma unroll
          for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int q = 0; q < 3; ++q)  // transpose of A(j, i)
              df_madd(acc[3 * k + r], wh[u][3 * q + r], wl[u][3 * q + r], x_h[q], x_l[q]);
        }
    }
  }
#pragma unroll
  for (int r = 0; r < 3 * K; ++r) sh[lane][r][slot] = acc[r];
  __syncthreads();
  for (int r = lane; r < 3 * K; r += W) {
    DF s = sh[0][r][slot];
#pragma unroll
    for (int u = 1; u < W; ++u) df_add(s, sh[u][r][slot].h, sh[u][r][slot].l);
    if (R.valid) {
      const size_t i = r * xs + R.row;
      y[i] = b[i] - ((double)s.h + (double)s.l);
    }
  }
}

// algorithmic bytes: stored values once (the transposed second read is meant
// to be an L2 hit by the launch order), x gathered once, y (and b) once
double sym3_bytes(const Sym3Op& so, int esz, int rows, int streams) {
  return (double)so.total * esz + (double)esz * 3.0 * rows * (1 + streams);
}

// one resident wave of a kernel walks the virtual blocks in plane order
template <class F> static int sym3_wave(F kernel, int block, int& w) {
  if (!w) {
    int dev = 0, sms = 0, occ = 0;
    SK_CUDA(cudaGetDevice(&dev));
    SK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    SK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, block, 0));
    w = std::max(1, sms * std::max(1, occ));
  }
  return w;
}

template <int W, int U>
static void sym3_launch_w(const Exec& ex, const Csr& m, const double* x, double* y, const double* b,
                          const DotScratch* ds, double* dot) {
  const Sym3Op& so = *m.sym;
  const Sym3Args a = sym3_args(so);
  const int nvb = sym3_blocks(so, a);
  if (nvb == 0) return;
  static thread_local int wave[2] = {};  // resident blocks per variant (dot or not)
  if (dot) {
    const int grid = std::min(nvb, sym3_wave(k_sym3<W, U, double, true>, 32 * W, wave[1]));
    SK_REQUIRE(ds && ds->fused_partial && grid <= ds->fused_cap, STOKES_ERR_ARG, "fused dot scratch too small");
    launch_dep(k_sym3<W, U, double, true>, grid, 32 * W, 0, ex, a, nvb, so.v64, x, (size_t)m.rows, b, y,
               ds->fused_partial, ds->fused_counter, dot);
  } else {
    const int grid = std::min(nvb, sym3_wave(k_sym3<W, U, double, false>, 32 * W, wave[0]));
    launch_dep(k_sym3<W, U, double, false>, grid, 32 * W, 0, ex, a, nvb, so.v64, x, (size_t)m.rows, b, y, nullptr,
               nullptr, nullptr);
  }
}

// four right-hand sides (x, y, b: [4][3][rows]): every stored block read once
// for the four
void sym3_launch4(const Exec& ex, const Csr& m, const double* x, double* y, const double* b) {
  const Sym3Op& so = *m.sym;
  const Sym3Args a = sym3_args(so);
  const int nvb = sym3_blocks(so, a);
  if (nvb == 0) return;
  static thread_local int wave = 0;
  const int grid = std::min(nvb, sym3_wave(k_sym3<4, 1, double, false, 4>, 128, wave));
  launch_dep(k_sym3<4, 1, double, false, 4>, grid, 128, 0, ex, a, nvb, so.v64, x, (size_t)m.rows, b, y, nullptr,
             nullptr, nullptr);
}

// Eight warps per 32 rows below 2^15 rows, four above: FP64 with the fused dot at
// 8^3 16.7 us against 20.9 for four (a thread per row: 45), at 24^3 100 against
// 104 for eight (148); the double-float residual at 48^3 298 us against 316 and
// 374 for eight (one, two entries in flight) and 321 for a thread per row.
constexpr int kSymWide = 1 << 15;

void sym3_launch(const Exec& ex, const Csr& m, const double* x, double* y, const double* b, const DotScratch* ds,
                 double* dot) {
  // entries in flight per warp lane: sym_batch (2 by default)
  const int u = m.sym->batch;
  if (m.rows < kSymWide) {
    if (u >= 4) sym3_launch_w<8, 4>(ex, m, x, y, b, ds, dot);
    else sym3_launch_w<8, 2>(ex, m, x, y, b, ds, dot);
  } else {
    if (u >= 4) sym3_launch_w<4, 4>(ex, m, x, y, b, ds, dot);
    else sym3_launch_w<4, 2>(ex, m, x, y, b, ds, dot);
  }
}

void sym3_residual_df(const Exec& ex, const Csr& m, const float* xh, const float* xl, const double* b, double* y) {
  const Sym3Op& so = *m.sym;
  const Sym3Args a = sym3_args(so);
  const int grid = sym3_blocks(so, a);
  if (grid == 0) return;
  if (m.rows < kSymWide)
    launch_dep(k_sym3_df<8, 2, 1>, grid, 256, 0, ex, a, so.v32, so.v32lo, xh, xl, (size_t)m.rows, b, y);
  else
    launch_dep(k_sym3_df<4, 2, 1>, grid, 128, 0, ex, a, so.v32, so.v32lo, xh, xl, (size_t)m.rows, b, y);
}

// four right-hand sides in one sweep (one entry in flight per lane)
void sym3_residual_df4(const Exec& ex, const Csr& m, const float* xh, const float* xl, const double* b, double* y) {
  const Sym3Op& so = *m.sym;
  const Sym3Args a = sym3_args(so);
  const int grid = sym3_blocks(so, a);
  if (grid == 0) return;
  launch_dep(k_sym3_df<4, 1, 4>, grid, 128, 0, ex, a, so.v32, so.v32lo, xh, xl, (size_t)m.rows, b, y);
}

}  // namespace sk
