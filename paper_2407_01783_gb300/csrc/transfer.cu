// FP32 P2 multigrid transfers without their matrices: the weights of a fine
// node are products of its barycentric coordinates in the coarse Kuhn mesh
// (logical positions), which are integers over a common denominator, so the
// kernels form them as exact small integers and divide the sum once.
#include <algorithm>

#include "internal.h"

namespace sk {

struct ProlongArgs {
  int mf, mc, nc, D;        // interior points per axis (fine, coarse); coarse cubes; denominator of the coordinates
  int step;                 // fine half-grid coordinate q sits at q step / D coarse cubes
  int total;                // fine interior nodes
  float inv;                // 1 / D^2
  FastDiv by_m, by_mm, by_D;
  SplitMap sm;
  int split;
};

// y += P x: a thread per fine node. Replaces CSR rows of 4.5 entries (8 bytes
// each, loaded before the gathers can start); bound by the latency of the gathers
// (L1 at 25%, DRAM at 5% at 36^3). us at
// 12^3, 25^3, 48^3, 64^3, 96^3: 2.7, 4.3, 14, 31, 103 (CSR 3.0, 5.8, 23, 67, 242).
// NR components: component-major, or
// node-interleaved (IL); the fine rows parity-split numbered if a.split.
template <int NR, bool IL>
__global__ void __launch_bounds__(256) k_prolong_p2(const ProlongArgs a, const float* __restrict__ x, size_t xs,
                                                   float* __restrict__ y, size_t ys) {
  dep_wait();
  const int t = blockIdx.x * 256 + threadIdx.x;
  if (t >= a.total) return;
  const int z = a.by_mm.div(t), tz = t - z * a.by_mm.d, yy = a.by_m.div(tz);
  const int q[3] = {tz - yy * a.by_m.d + 1, yy + 1, z + 1};
  int b[3], r[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int p = q[c] * a.step;
    b[c] = a.by_D.div(p);  // below nc: q is interior
    r[c] = p - b[c] * a.D;
  }
  // axes by decreasing local coordinate (the order of equal ones is immaterial:
  // the vertex between them has weight 0)
  const int s[3] = {1, a.mc, a.mc * a.mc};
  int r0 = r[0], r1 = r[1], r2 = r[2], b0 = 1, b1 = 2, b2 = 4, s0 = s[0], s1 = s[1], s2 = s[2];
  auto order = [](int& ra, int& rb, int& ba, int& bb, int& sa, int& sb) {
    if (rb > ra) {
      int u = ra; ra = rb; rb = u;
      u = ba; ba = bb; bb = u;
      u = sa; sa = sb; sb = u;
    }
  };
  order(r0, r1, b0, b1, s0, s1);
  order(r1, r2, b1, b2, s1, s2);
  order(r0, r1, b0, b1, s0, s1);
  const int l[4] = {a.D - r0, r0 - r1, r1 - r2, r2};                    // coordinates times D
  const int off[4] = {0, s0, s0 + s1, s0 + s1 + s2};                    // vertex offsets (half a half-grid step)
  const int bits[4] = {0, b0, b0 | b1, 7};
  // coarse faces touched on the boundary: node on them carries no unknown
  int lo = 0, hi = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) lo |= (b[c] == 0) << c, hi |= (b[c] == a.nc - 1) << c;
  const int base = (2 * b[0] - 1) + s[1] * (2 * b[1] - 1) + s[2] * (2 * b[2] - 1);
  // weights times D^2 and columns (-1: no unknown or weight 0), then all loads
  // together, then the sums
  float w[10];
  int at[10];
  int e = 0;
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = u; v < 4; ++v, ++e) {
      const int num = u == v ? l[u] * (2 * l[u] - a.D) : 4 * l[u] * l[v];
      const bool out = num == 0 || (lo & ~(bits[u] | bits[v])) || (hi & (bits[u] & bits[v]));
      w[e] = out ? 0.f : (float)num;
      at[e] = out ? -1 : base + off[u] + off[v];
    }
  const size_t row = a.split ? (size_t)a.sm(t) : (size_t)t;
  if constexpr (IL) {
#pragma unroll
    for (int k = 0; k < NR / 4; ++k) {
      float4 v[10];
#pragma unroll
      for (int i = 0; i < 10; ++i)
        v[i] = at[i] >= 0 ? reinterpret_cast<const float4*>(x)[(size_t)at[i] * (NR / 4) + k]
                          : make_float4(0.f, 0.f, 0.f, 0.f);
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < 10; ++i) s.x += w[i] * v[i].x, s.y += w[i] * v[i].y, s.z += w[i] * v[i].z, s.w += w[i] * v[i].w;
      float4& o = reinterpret_cast<float4*>(y)[row * (NR / 4) + k];
      float4 r = o;
      r.x += a.inv * s.x, r.y += a.inv * s.y, r.z += a.inv * s.z, r.w += a.inv * s.w;
      o = r;
    }
  } else {
    float v[10][NR];
#pragma unroll
    for (int i = 0; i < 10; ++i)
#pragma unroll
      for (int k = 0; k < NR; ++k) v[i][k] = at[i] >= 0 ? x[k * xs + at[i]] : 0.f;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < 10; ++i) s += w[i] * v[i][k];
      y[k * ys + row] += a.inv * s;
    }
  }
}

static int gcd_of(int a, int b) { return b ? gcd_of(b, a % b) : a; }

void prolong_p2(const Exec& ex, int nf, int nc, int nr, const float* x, float* y, bool il, const SplitMap* sm) {
  const int g = gcd_of(nc, 2 * nf);
  const int mf = 2 * nf - 1, mc = 2 * nc - 1, D = 2 * nf / g;
  ProlongArgs a{mf, mc, nc, D, nc / g, mf * mf * mf, 1.f / ((float)D * (float)D), FastDiv(mf), FastDiv(mf * mf),
                FastDiv(D), sm ? *sm : SplitMap{}, sm ? 1 : 0};
  const int grid = cdiv(a.total, 256);
  const size_t xs = (size_t)mc * mc * mc, ys = (size_t)a.total;
  if (nr == 3 && !il) launch_dep(k_prolong_p2<3, false>, grid, 256, 0, ex, a, x, xs, y, ys);
  else if (nr == 12 && il) launch_dep(k_prolong_p2<12, true>, grid, 256, 0, ex, a, x, xs, y, ys);
  else throw Error(STOKES_ERR_ARG, "P2 transfer: 3 component-major or 12 interleaved components");
  SK_CHECK_LAUNCH();
}

// Restriction on nested meshes (nf = 2 nc): the fine nodes q = 2 Q + d around a
// coarse node Q and their weights depend on Q's parity class only.
constexpr int kRestrictMax = 290;  // entries of all classes
struct RestrictArgs {
  int mf = 0, mc = 0, nc = 0, beg[9] = {};
  FastDiv by_o{1}, by_e{1};
  int lin[kRestrictMax];    // offset of fine node 2 Q + d from 2 Q
  float w[kRestrictMax];    // weight times 16
  signed char dx[kRestrictMax];  // x offset (parity-split numbering)
  SplitMap sm;
  int split = 0;
};

// offsets d and weights (times 16) by class, the same for every mesh
struct RestrictTable {
  int n = 0, beg[9] = {};
  signed char d[kRestrictMax][3];
  float w[kRestrictMax];
  RestrictTable() {
    for (int c = 0; c < 8; ++c) {
      beg[c] = n;
      const int Q[3] = {4 + (c & 1), 4 + ((c >> 1) & 1), 4 + (c >> 2)};
      for (int z = -3; z <= 3; ++z)
        for (int y = -3; y <= 3; ++y)
          for (int x = -3; x <= 3; ++x) add(Q, x, y, z);
    }
    beg[8] = n;
  }
  void add(const int* Q, int x, int y, int z) {
    const int q[3] = {2 * Q[0] + x, 2 * Q[1] + y, 2 * Q[2] + z};
    int b[3], r[3], p[3] = {0, 1, 2};
    for (int k = 0; k < 3; ++k) b[k] = q[k] / 4, r[k] = q[k] % 4;
    std::stable_sort(p, p + 3, [&](int i, int j) { return r[i] > r[j]; });
    const int l[4] = {4 - r[p[0]], r[p[0]] - r[p[1]], r[p[1]] - r[p[2]], r[p[2]]};
    int v[4][3];
    for (int k = 0; k < 4; ++k)
      for (int i = 0; i < 3; ++i) v[k][i] = b[i];
    for (int k = 1; k < 4; ++k)
      for (int i = k; i < 4; ++i) ++v[i][p[k - 1]];
    int num = 0;
    for (int i = 0; i < 4; ++i)
      for (int j = i; j < 4; ++j)
        if (v[i][0] + v[j][0] == Q[0] && v[i][1] + v[j][1] == Q[1] && v[i][2] + v[j][2] == Q[2])
          num += i == j ? l[i] * (2 * l[i] - 4) : 4 * l[i] * l[j];
    if (!num) return;
    SK_REQUIRE(n < kRestrictMax, STOKES_ERR_ARG, "restriction table overflow");
    d[n][0] = (signed char)x, d[n][1] = (signed char)y, d[n][2] = (signed char)z;
    w[n++] = (float)num;
  }
};

static RestrictArgs restrict_args(int nc) {
  static const RestrictTable t;
  RestrictArgs a;
  a.by_o = FastDiv(nc);
  a.by_e = FastDiv(std::max(1, nc - 1));
  a.nc = nc;
  a.mc = 2 * nc - 1;
  a.mf = 4 * nc - 1;
  for (int c = 0; c < 9; ++c) a.beg[c] = t.beg[c];
  for (int e = 0; e < t.n; ++e) {
    a.lin[e] = t.d[e][0] + a.mf * (t.d[e][1] + a.mf * t.d[e][2]);
    a.dx[e] = t.d[e][0];
    a.w[e] = t.w[e];
  }
  return a;
}

// y = R x: 32 coarse nodes of one class (blockIdx.y) and, component-major, one
// component (blockIdx.z) per block; the entries of a node are spread over the
// block's eight warps (a coarse vertex has 125, the other classes 19 or 27).
// Interleaved: a lane handles four of the NR components of a node.
template <int NR, bool IL>
__global__ void __launch_bounds__(256) k_restrict_p2(const RestrictArgs a, const float* __restrict__ x, size_t xs,
                                                    float* __restrict__ y, size_t ys) {
  dep_wait();
  constexpr int L = IL ? NR / 4 : 1;  // lanes per node
  using V = typename std::conditional<IL, float4, float>::type;
  __shared__ V sh[8][32];
  const int c = blockIdx.y, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int odd[3] = {c & 1, (c >> 1) & 1, c >> 2};
  const int ex = a.nc - 1 + odd[0], ey = a.nc - 1 + odd[1], ez = a.nc - 1 + odd[2];
  const int g = blockIdx.x * 32 + lane, t = g / L, part = g % L;
  const bool live = t < ex * ey * ez;
  const int tt = live ? t : 0;
  const int lines = (odd[0] ? a.by_o : a.by_e).div(tt), kz = (odd[1] ? a.by_o : a.by_e).div(lines);  // by nc, nc - 1
  const int Qx = 2 - odd[0] + 2 * (tt - lines * ex), Qy = 2 - odd[1] + 2 * (lines - kz * ey), Qz = 2 - odd[2] + 2 * kz;
  const int base = (2 * Qx - 1) + a.mf * ((2 * Qy - 1) + a.mf * (2 * Qz - 1));  // fine node 2 Q
  const int line = base - (2 * Qx - 1);
  V s;
  if constexpr (IL) s = make_float4(0.f, 0.f, 0.f, 0.f);
  else s = 0.f;
  const int e1 = a.beg[c + 1];
#pragma unroll 4
  for (int e = a.beg[c] + w; e < e1; e += 8) {
    // every fine node with a weight is an interior one: the coarse basis
    // function of an interior node vanishes on the boundary
    size_t at;
    if (a.split) {
      const int i = 2 * Qx - 1 + a.dx[e];
      at = (size_t)(line + a.lin[e] - a.dx[e] + ((i & 1) ? a.sm.half + (i >> 1) : (i >> 1)));
    } else {
      at = (size_t)(base + a.lin[e]);
    }
    const float f = a.w[e];
    if constexpr (IL) {
      const float4 v = reinterpret_cast<const float4*>(x)[at * L + part];
      s.x += f * v.x, s.y += f * v.y, s.z += f * v.z, s.w += f * v.w;
    } else {
      s += f * x[blockIdx.z * xs + at];
    }
  }
  sh[w][lane] = s;
  __syncthreads();
  if (w || !live) return;
  const size_t row = (size_t)(Qx - 1) + (size_t)a.mc * ((Qy - 1) + (size_t)a.mc * (Qz - 1));
  constexpr float inv = 1.f / 16.f;
  auto sum = [&](auto get) {
    return inv * (((get(sh[0][lane]) + get(sh[1][lane])) + (get(sh[2][lane]) + get(sh[3][lane]))) +
                  ((get(sh[4][lane]) + get(sh[5][lane])) + (get(sh[6][lane]) + get(sh[7][lane]))));
  };
  if constexpr (IL)
    reinterpret_cast<float4*>(y)[row * L + part] =
        make_float4(sum([](const V& v) { return v.x; }), sum([](const V& v) { return v.y; }),
                    sum([](const V& v) { return v.z; }), sum([](const V& v) { return v.w; }));
  else
    y[blockIdx.z * ys + row] = sum([](const V& v) { return v; });
}

// Nested levels only. Component-major gathers are 4 words apart in x: above 32
// cubes the CSR product (several lanes per row) is faster, below it its index
// loads cost more than the gathers. us at 8^3, 24^3, 40^3, 48^3: 2.9, 3.9, 10.3,
// 16.2 against 3.3, 4.5, 9.1, 13.7. Interleaved rows are contiguous: always.
bool restrict_p2_fits(int nf, int nc, bool il) { return nf == 2 * nc && (il || nf <= 32); }

void restrict_p2(const Exec& ex, int nc, int nr, const float* x, float* y, bool il, const SplitMap* sm) {
  RestrictArgs a = restrict_args(nc);
  a.split = sm ? 1 : 0;
  if (sm) a.sm = *sm;
  const size_t xs = (size_t)a.mf * a.mf * a.mf, ys = (size_t)a.mc * a.mc * a.mc;
  const int rows = nc * nc * nc;  // most of any class
  if (nr == 3 && !il) launch_dep(k_restrict_p2<3, false>, dim3(cdiv(rows, 32), 8, 3), 256, 0, ex, a, x, xs, y, ys);
  else if (nr == 12 && il)
    launch_dep(k_restrict_p2<12, true>, dim3(cdiv(3LL * rows, 32), 8), 256, 0, ex, a, x, xs, y, ys);
  else throw Error(STOKES_ERR_ARG, "P2 transfer: 3 component-major or 12 interleaved components");
  SK_CHECK_LAUNCH();
}

}  // namespace sk
