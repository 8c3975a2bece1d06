// Small lattices iterated on chip, with every relaxation time 1: a CTA - or a cluster of up to
// eight, each with a share of the rows - holds a lattice's state in registers and takes step
// after step on it without touching global memory (arXiv 2301.12869, Sec. III; the physics and
// the three-number state (drho, j_x, j_y): lbm_unit.cuh).
//
// The general batch kernel reads each node's nine values twice a step from L2 and stores nine; its
// steps are bound by that latency. Here FP32 steps are bound by a thread's dependency chain (1.3
// us a step for one column of 128 rows, 2.7 us for 1024 columns, 7 an SM), double-float by the
// instruction issue (about 1100 a node), FP64 by the SM's FP64 pipe.
//
// Layout: a thread holds Q neighbouring nodes of a row (4 FP32 nodes as two packed pairs; one
// FP64 or double-float node, whose arithmetic is the bound and wants the most warps), up to R
// such items; a row takes 2^row_log2 lanes of a warp, so x neighbours (periodic) come by
// shuffles. y neighbours go through shared memory, once for the potential's stencil sums
//   A = psi_x difference / 12, B = psi/3 + (psi(x-1) + psi(x+1))/12  (double-float: 3 sqrt(3) times)
//   S_x = 4 A(y) + A(y+1) + A(y-1),  S_y = B(y+1) - B(y-1)
// and once for what a node sends up (u1 = f2 + f5(x-1) + f6(x+1), u2 = f5(x-1) - f6(x+1)) and
// down (v1, v2 of f4, f8, f7). Two barriers a step; a cluster's CTAs write their edge rows into
// their neighbours' halo rows (distributed shared memory) and use the cluster's barrier.
// <rho> of Eq. Gravity_2 is the sum of drho: warp totals, exchanged with the second barrier of
// a step and added by every warp after the first of the next. FP32 and double-float sums are pairs (48
// bits, the FP64 pipe left alone): double-float columns of both forms are 8.3e-16 rms from 80 bits after 300
// steps, 8.1e-16 between wet walls, where <rho> also sets the wall density; with FP64 sums in the
// general kernel 1.7e-15 and 1.7e-15.
//
// The populations are read at the start of a run (pulled into M_0) and written by the last
// step, whose collision forms them.
#pragma once

#include "lbm_column.h"
#include "lbm_dd.cuh"
#include "lbm_lane.cuh"
#include "lbm_ptx.cuh"
#include "lbm_unit.cuh"

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cfloat>
#include <cmath>
#include <cstdint>

namespace lbm {

template <typename T>
struct ItemOf;
template <>
struct ItemOf<float> {
  using V = f2;
  using S = dd;  // sums of drho
  using M = dd;  // largest change
  static constexpr int N = 2, Q = 4, max_threads = 256;
};
template <>
struct ItemOf<double> {
  using V = double;
  using S = double;
  using M = double;
  static constexpr int N = 1, Q = 1, max_threads = 256;
};
template <>
struct ItemOf<dd> {
  using V = dd;
  using S = dd;
  using M = dd;
  static constexpr int N = 1, Q = 1, max_threads = 256;
};

constexpr int kColWarps = 8;    // most warps of a CTA
constexpr int kColCluster = 8;   // most CTAs of a cluster (the portable size)

namespace {

// the real type's conversions to the arithmetic type
template <typename V>
__device__ __forceinline__ V real(double c);
template <>
__device__ __forceinline__ f2 real<f2>(double c) { return make_f2(float(c), float(c)); }
template <>
__device__ __forceinline__ double real<double>(double c) { return c; }
template <>
__device__ __forceinline__ dd real<dd>(double c) { return dd_of(c); }

// Double-float columns hold sqrt(3) psi, and its stencil sums without their factor 1/3: psi^2 then has
// no constant that is a third (3 k_2, 3 k_3 are exact for the usual a, G), and the force takes -G/9 and
// the sigma term 1/27. The double-float 1/3 is 2^-50 too small at every step alike: over 300 steps of
// 384 columns of 64 rows the populations' error against FP64 was 5.1e-14 with it, and is 3.0e-14 (4.3e-14
// in the order of lbm_physics.cuh, which has it too but rounds differently); two products a node less.
template <typename V>
constexpr double kPsi2 = 1.0;  // the square of the factor
template <>
constexpr double kPsi2<dd> = 3.0;

template <typename V>
__device__ UnitT<V> column_unit(const ColumnArgs& a, const BatchCol& c) {
  constexpr double s = kPsi2<V>;
  UnitT<V> u{};
  u.p.rho_ref = real<V>(c.rho_ref);
  u.p.RT = real<V>(c.RT);
  u.p.a = real<V>(a.a);
  u.p.b4 = real<V>(a.b / 4.0);
  u.p.twoOverG = real<V>(2.0 / a.G);
  u.p.negG = real<V>(-a.G / (s * s));
  u.p.gx = real<V>(c.gx);
  u.p.gy = real<V>(c.gy);
  u.p.form = c.form;
  u.k1 = real<V>(2.0 * s * c.RT / a.G);
  u.p.k2 = real<V>(-2.0 * s * a.a / a.G);
  u.p.k3 = real<V>(s == 3.0 ? -2.0 / a.G : -2.0 / (3.0 * a.G));
  u.p.kS = real<V>(a.G * a.G * a.sig_e / (72.0 * s * s * s));
  return u;
}

// ---- an item's nodes in global memory. The four nodes of an FP32 item are paired (0, 2) and
// (1, 3): a pair's neighbours on one side are the other pair, and on the other side that pair
// with its halves exchanged, one of them from the next item
__device__ __forceinline__ Lane<f2, 2> load_item(const float* p) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  return {{make_f2(q.x, q.z), make_f2(q.y, q.w)}};
}
__device__ __forceinline__ Lane<double, 1> load_item(const double* p) { return {{*p}}; }
__device__ __forceinline__ Lane<dd, 1> load_item(const dd* p) {
  const float2 q = *reinterpret_cast<const float2*>(p);
  return {{dd{q.x, q.y}}};
}
__device__ __forceinline__ void store_item(float* p, const Lane<f2, 2>& q) {
  *reinterpret_cast<float4*>(p) = make_float4(lo(q.v[0]), lo(q.v[1]), hi(q.v[0]), hi(q.v[1]));
}
__device__ __forceinline__ void store_item(double* p, const Lane<double, 1>& q) { *p = q.v[0]; }
__device__ __forceinline__ void store_item(dd* p, const Lane<dd, 1>& q) {
  *reinterpret_cast<float2*>(p) = make_float2(q.v[0].hi, q.v[0].lo);
}

template <class Get>
__device__ __forceinline__ Lane<f2, 2> item_left(const Lane<f2, 2>& q, Get get) {  // value at x - 1
  return {{make_f2(get(hi(q.v[1])), lo(q.v[1])), q.v[0]}};
}
template <class Get>
__device__ __forceinline__ Lane<f2, 2> item_right(const Lane<f2, 2>& q, Get get) {  // value at x + 1
  return {{q.v[1], make_f2(hi(q.v[0]), get(lo(q.v[0])))}};
}
template <typename V, class Get>
__device__ __forceinline__ Lane<V, 1> item_left(const Lane<V, 1>& q, Get get) {
  return {{get(q.v[0])}};
}
template <typename V, class Get>
__device__ __forceinline__ Lane<V, 1> item_right(const Lane<V, 1>& q, Get get) {
  return {{get(q.v[0])}};
}

// ---- an item's mass, totals over a warp
__device__ __forceinline__ dd item_mass(const Lane<f2, 2>& q) {
  return dd_two_sum(lo(q.v[0]), hi(q.v[0])) + dd_two_sum(lo(q.v[1]), hi(q.v[1]));
}
__device__ __forceinline__ double item_mass(const Lane<double, 1>& q) { return q.v[0]; }
__device__ __forceinline__ dd item_mass(const Lane<dd, 1>& q) { return q.v[0]; }
// sum over groups of `width` lanes (a power of two), in every lane
template <typename S>
__device__ __forceinline__ S lanes_total(S s, int width) {
  const int lane = threadIdx.x & 31;
  for (int m = width >> 1; m; m >>= 1) s = s + lane_value(s, lane ^ m);
  return s;
}

template <typename S>
__device__ __forceinline__ S mass_of(double v);
template <>
__device__ __forceinline__ dd mass_of<dd>(double v) { return dd_of(v); }
template <>
__device__ __forceinline__ double mass_of<double>(double v) { return v; }
template <typename V, typename S>
__device__ __forceinline__ V mean_value(S s);
template <>
__device__ __forceinline__ f2 mean_value<f2, dd>(dd s) { return make_f2(s.hi, s.hi); }
template <>
__device__ __forceinline__ double mean_value<double, double>(double s) { return s; }
template <>
__device__ __forceinline__ dd mean_value<dd, dd>(dd s) { return s; }
// node j of an item as a double
__device__ __forceinline__ double hsum_node(const Lane<f2, 2>& q, int j) {
  const f2 p = q.v[j & 1];
  return double((j >> 1) ? hi(p) : lo(p));
}
__device__ __forceinline__ double hsum_node(const Lane<double, 1>& q, int) { return q.v[0]; }
__device__ __forceinline__ double hsum_node(const Lane<dd, 1>& q, int) { return hsum(q.v[0]); }

// the item's low parts: zero but for FP32, whose densities a residual compares beyond FP32
template <typename V, int N>
__device__ __forceinline__ Lane<V, N> two_sum_error(const Lane<V, N>& a, const Lane<V, N>& b, const Lane<V, N>& s) {
  const Lane<V, N> bb = s - a;
  return (a - (s - bb)) + (b - bb);
}

// the larger of m and d; a NaN d does not count
__device__ __forceinline__ dd larger(dd m, dd d) { return d.hi > m.hi || (d.hi == m.hi && d.lo > m.lo) ? d : m; }
__device__ __forceinline__ double larger(double m, double d) { return fmax(m, d); }
__device__ __forceinline__ dd magnitude(dd d) { return d.hi < 0.f ? -d : d; }
// |(a + al) - (b + bl)|: the difference of the values is exact, so the pair is good to 2^-24 of the
// change beyond what the low parts hold
__device__ __forceinline__ dd change(float a, float al, float b, float bl) {
  const dd s = dd_two_sum(a, -b);
  if (!(fabsf(s.hi) <= FLT_MAX)) return dd{fabsf(s.hi), 0.f};  // infinite: no error terms
  return magnitude(dd_two_sum(s.hi, __fadd_rn(s.lo, __fsub_rn(al, bl))));
}

// largest |rho - previous rho| of an item from (value, low part) pairs, as a pair: it decides
// convergence and is the caller's residual in FP64 (the FP64 pipe is left to FP64 columns)
__device__ __forceinline__ dd item_change(const Lane<f2, 2>& a, const Lane<f2, 2>& al, const Lane<f2, 2>& b,
                                          const Lane<f2, 2>& bl) {
  dd m{};
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    m = larger(m, change(lo(a.v[j]), lo(al.v[j]), lo(b.v[j]), lo(bl.v[j])));
    m = larger(m, change(hi(a.v[j]), hi(al.v[j]), hi(b.v[j]), hi(bl.v[j])));
  }
  return m;
}
__device__ __forceinline__ double item_change(const Lane<double, 1>& a, const Lane<double, 1>&,
                                              const Lane<double, 1>& b, const Lane<double, 1>&) {
  return fmax(0.0, fabs(a.v[0] - b.v[0]));
}
__device__ __forceinline__ dd item_change(const Lane<dd, 1>& a, const Lane<dd, 1>&, const Lane<dd, 1>& b,
                                          const Lane<dd, 1>&) {
  return larger(dd{}, change(a.v[0].hi, a.v[0].lo, b.v[0].hi, b.v[0].lo));
}

// pull streaming (Eq. LBE) of node (x, y): the nine populations arriving there
template <typename T>
__device__ __forceinline__ void pull_node(const T* f, int nx, int ny, size_t N, int x, int y, T (&g)[9]) {
  const int xl = x == 0 ? nx - 1 : x - 1, xr = x == nx - 1 ? 0 : x + 1;
  const size_t row = size_t(y) * nx, node = row + x;
  const bool lo_w = y == 0, hi_w = y == ny - 1;
  g[0] = f[node];
  g[1] = f[1 * N + row + xl];
  g[3] = f[3 * N + row + xr];
  g[2] = lo_w ? f[4 * N + node] : f[2 * N + row - nx + x];
  g[5] = lo_w ? f[7 * N + node] : f[5 * N + row - nx + xl];
  g[6] = lo_w ? f[8 * N + node] : f[6 * N + row - nx + xr];
  g[4] = hi_w ? f[2 * N + node] : f[4 * N + row + nx + x];
  g[7] = hi_w ? f[5 * N + node] : f[7 * N + row + nx + xr];
  g[8] = hi_w ? f[6 * N + node] : f[8 * N + row + nx + xl];
}
// moments of a node's pulled populations in the type A; k_lo, k_hi: Zou-He's K at the bottom, top
template <typename A>
struct Pulled {
  A dr, jx, jy, k_lo, k_hi;
};
template <typename A, typename T>
__device__ __forceinline__ Pulled<A> pulled_moments(const T* f, int nx, int ny, size_t N, int x, int y) {
  T g[9];
  pull_node(f, nx, ny, N, x, y, g);
  A d[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) d[i] = A(g[i]);
  const A h = d[0] + (d[1] + d[3]), up = d[2] + (d[5] + d[6]), dn = d[4] + (d[7] + d[8]);
  return {h + (up + dn), (d[1] - d[3]) + ((d[5] - d[7]) - (d[6] - d[8])), up - dn, h + (dn + dn), h + (up + up)};
}
template <typename T>
__device__ __forceinline__ double stored_mass(const T* f, size_t N, size_t n) {
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < 9; ++i) s += hsum(f[i * N + n]);
  return s;
}
__device__ __forceinline__ void set_node(Lane<f2, 2>& q, int j, float v) {
  f2& p = q.v[j & 1];
  p = (j >> 1) ? make_f2(lo(p), v) : make_f2(v, hi(p));
}
__device__ __forceinline__ void set_node(Lane<f2, 2>& q, int j, double v) { set_node(q, j, float(v)); }
__device__ __forceinline__ void set_node(Lane<double, 1>& q, int, double v) { q.v[0] = v; }
__device__ __forceinline__ void set_node(Lane<dd, 1>& q, int, dd v) { q.v[0] = v; }
__device__ __forceinline__ void set_node(Lane<dd, 1>& q, int, double v) { q.v[0] = dd_of(v); }
// the extrapolation's weights from the packed Gram matrix g of the differences: c (c_kMpeK = 1)
// minimising |sum_j c_j u_j| by Gaussian elimination with partial pivoting, gam = c / sum c
__device__ inline bool mpe_solve(const double* g, double* gam) {
  constexpr int NU = kMpeK + 1;
  auto at = [&](int i, int j) {
    if (i > j) {
      const int t = i;
      i = j;
      j = t;
    }
    return g[i * NU - i * (i - 1) / 2 + (j - i)];
  };
  double Am[kMpeK][kMpeK + 1];  // sum_{j<K} G_ij c_j = -G_iK for i < K
  for (int i = 0; i < kMpeK; ++i) {
    for (int j = 0; j < kMpeK; ++j) Am[i][j] = at(i, j);
    Am[i][kMpeK] = -at(i, kMpeK);
  }
  bool ok = at(kMpeK, kMpeK) > 0.0;
  const double scale = at(0, 0) + at(kMpeK, kMpeK);
  for (int ci = 0; ci < kMpeK && ok; ++ci) {
    int piv = ci;
    for (int i = ci + 1; i < kMpeK; ++i)
      if (fabs(Am[i][ci]) > fabs(Am[piv][ci])) piv = i;
    if (!(fabs(Am[piv][ci]) > 1e-14 * scale)) {
      ok = false;
      break;
    }
    if (piv != ci)
      for (int j = 0; j <= kMpeK; ++j) {
        const double t = Am[ci][j];
        Am[ci][j] = Am[piv][j];
        Am[piv][j] = t;
      }
    for (int i = ci + 1; i < kMpeK; ++i) {
      const double f = Am[i][ci] / Am[ci][ci];
      for (int j = ci; j <= kMpeK; ++j) Am[i][j] -= f * Am[ci][j];
    }
  }
  double c[NU];
  c[kMpeK] = 1.0;
  for (int i = kMpeK - 1; i >= 0 && ok; --i) {
    double sum = Am[i][kMpeK];
    for (int j = i + 1; j < kMpeK; ++j) sum -= Am[i][j] * c[j];
    c[i] = sum / Am[i][i];
  }
  double S = 0.0, Sabs = 0.0;
  for (int j = 0; j < NU && ok; ++j) {
    S += c[j];
    Sabs += fabs(c[j]);
  }
  ok = ok && isfinite(S) && fabs(S) > 1e-8 * Sabs;
  for (int j = 0; j < NU; ++j) gam[j] = ok ? c[j] / S : 0.0;
  return ok;
}

// ALONE: a row is one lane, its own neighbour on both sides (four FP32 columns)
template <typename T, int R, bool ACC, bool ALONE>
__global__ void __launch_bounds__(ItemOf<T>::max_threads, sizeof(T) == 4 && R > 1 ? 1 : 2)
    column_kernel(const __grid_constant__ ColumnArgs a) {
  namespace cg = cooperative_groups;
  using V = typename ItemOf<T>::V;
  using S = typename ItemOf<T>::S;
  using M = typename ItemOf<T>::M;
  constexpr int N = ItemOf<T>::N, Q = ItemOf<T>::Q;
  constexpr bool LOW = sizeof(T) == 4;  // FP32: densities beyond FP32 for the residual
  using L = Lane<V, N>;
  constexpr int NU = kMpeK + 1, NG = NU * (NU + 1) / 2;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ S mass_s[kColCluster * kColWarps];
  __shared__ M max_s[kColCluster * kColWarps];
  __shared__ double gram_s[ACC ? NG : 1][ACC ? kColCluster * kColWarps : 1];
  __shared__ double gam_s[NU];
  __shared__ int col_s, ok_s, bad_s[kColCluster];
  // the column's constants: double-float and FP64 ones in shared memory, where they leave registers to
  // the arithmetic's chains (whole calls: 1024 columns double-float 13.1 -> 12.3 ms, 320 columns FP64
  // 17.3 -> 16.8 ms; 4 x 200 FP64 4.70 -> 4.60 us a step). FP32 ones cost its chain a load: 5.84 -> 5.95 ms
  constexpr bool SHARED_K = sizeof(T) == 8;
  __shared__ UnitT<V> k_s;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x, NW = NT >> 5;
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = a.cluster, rank = cs > 1 ? int(cluster.block_rank()) : 0;
  const int P = 1 << a.row_log2, nx = a.nx, m = nx / Q;
  const int l = lane & (P - 1), base = lane & ~(P - 1);
  const int src_l = base + (l == 0 ? m - 1 : l - 1), src_r = base + (l + 1 >= m ? 0 : l + 1);
  const RunParams run = a.run ? *a.run : a.run_one;
  const int K = run.check_every;

  // shared rows: [-1, rows] of each array
  const int cap = (a.rows_cap + 2) * P;
  L* sA = reinterpret_cast<L*>(sm_raw);
  L* sB = sA + cap;
  L* su1 = sB + cap;
  L* su2 = su1 + cap;
  L* sv1 = su2 + cap;
  L* sv2 = sv1 + cap;
  L* sul = LOW ? sv2 + cap : sv2;  // low parts of u1, v1
  L* svl = LOW ? sul + cap : sv2;
  auto remote = [&](L* p, int r) { return cluster.map_shared_rank(p, r); };
  auto sync = [&] {
    if (cs > 1)
      cluster.sync();
    else
      __syncthreads();
  };
  auto left = [&](const L& q) { return item_left(q, [&](auto v) { return ALONE ? v : lane_value(v, src_l); }); };
  auto right = [&](const L& q) { return item_right(q, [&](auto v) { return ALONE ? v : lane_value(v, src_r); }); };
  const V zero = cst<V>(0.0);
  const L zeroL = splat_lane<V, N>(zero);

  for (int turn = 0;; ++turn) {
    // ---- take a column (work stealing by rank 0, or the one lattice)
    int c = 0;
    BatchCol col;
    if (a.order) {
      sync();
      if (rank == 0 && tid == 0) {
        const int ci = atomicAdd(a.counter, 1);
        for (int r = 0; r < cs; ++r) *(cs > 1 ? cluster.map_shared_rank(&col_s, r) : &col_s) = ci;
      }
      sync();
      if (col_s >= a.ncols) break;
      c = a.order[col_s];
      col = a.cols[c];
    } else {
      if (turn) break;
      col = a.one;
    }
    UnitT<V> k_r{};
    if constexpr (!SHARED_K)
      k_r = column_unit<V>(a, col);
    else if (tid == 0)
      k_s = column_unit<V>(a, col);
    const UnitT<V>& k = SHARED_K ? k_s : k_r;
    const long long t_start = [] { long long t; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)); return t; }();
    const int ny = col.ny;
    const size_t NN = size_t(nx) * ny;
    const int rbase = ny / cs, rrem = ny - rbase * cs;
    const int rows = rbase + (rank < rrem ? 1 : 0), y0 = rank * rbase + min(rank, rrem);
    const int rows_dn = rank > 0 ? rbase + (rank - 1 < rrem ? 1 : 0) : 0;  // rows of the rank below
    const int items = rows * P;
    const bool mean = col.form == 2, zh = a.zh != 0;
    const S inv_n = mass_of<S>(1.0 / double(NN));
    T* f = static_cast<T*>(a.f) + 9 * col.node_off;
    T* prev = static_cast<T*>(a.scratch) + 9 * col.node_off;  // compared density: [0, N), low part [N, 2N)

    // ---- this thread's items: local index i, row r, node index n; halo rows beyond the walls are zero
    auto item = [&](int q) { return tid + q * NT; };
    auto warp_live = [&](int q) { return 32 * warp + q * NT < items; };  // uniform over the warp
    auto live = [&](int q) { return item(q) < items && l < m; };
    if (tid < P) {
      const int top = (rows + 1) * P + tid;
      if (rank == 0) su1[tid] = su2[tid] = zeroL;
      if (rank == cs - 1) sv1[top] = sv2[top] = zeroL;
      if (LOW && rank == 0) sul[tid] = zeroL;
      if (LOW && rank == cs - 1) svl[top] = zeroL;
    }
    // every rank's warp totals to every rank
    auto put_mass = [&](S s) {
      s = lanes_total(s, 32);
      if (lane < cs) {
        S* dst = &mass_s[rank * NW + warp];
        *(cs > 1 ? cluster.map_shared_rank(dst, lane) : dst) = s;
      }
    };
    auto mean_of_mass = [&] {
      const int n = cs * NW;
      int w = 1;
      while (w < min(n, 32)) w <<= 1;
      S s{};
      for (int q = lane & (w - 1); q < n; q += w) s = s + mass_s[q];
      return lanes_total(s, w) * inv_n;  // <rho> - rho_ref
    };

    // ---- M_0: the moments of the stored populations, pulled; FP32 columns that are checked in
    // their first step also hold what FP32 does not of the density
    const bool low_first = LOW && K == 2;
    L dr[R], jx[R], jy[R], dl[R], Kq[R];
    double kx[LOW ? R * Q : 1];
    double mass0 = 0.0;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      dr[q] = jx[q] = jy[q] = dl[q] = Kq[q] = zeroL;
      if (live(q)) {
        const int y = y0 + (item(q) >> a.row_log2);
#pragma unroll
        for (int j = 0; j < Q; ++j) {
          const int x = l * Q + j;
          const auto g = pulled_moments<T>(f, nx, ny, NN, x, y);
          set_node(dr[q], j, g.dr);
          set_node(jx[q], j, g.jx);
          set_node(jy[q], j, g.jy);
          set_node(Kq[q], j, y == 0 ? g.k_lo : g.k_hi);
          if (zh && mean) mass0 += stored_mass(f, NN, size_t(y) * nx + x);
          if constexpr (LOW) {
            if (low_first) {
              const auto e = pulled_moments<double>(f, nx, ny, NN, x, y);
              set_node(dl[q], j, e.dr - double(g.dr));
              kx[q * Q + j] = y == 0 ? e.k_lo : e.k_hi;
            }
          }
        }
      }
    }
    S zmean{};  // Zou-He: <rho> - rho_ref of the collision of the current moments
    auto closure = [&](L (&Kq)[R], S mc, bool low, const double* kexact) {
      // wall-row items: dr, j from K with <rho> - rho_ref = mc
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int y = y0 + (item(q) >> a.row_log2);
        if (live(q) && (y == 0 || y == ny - 1)) {
#pragma unroll
          for (int j = 0; j < N; ++j)
            unit_zou_he(Kq[q].v[j], y == 0, mean_value<V>(mc), k, dr[q].v[j], jx[q].v[j], jy[q].v[j]);
          if (LOW && low) {
            const double sg = (y == 0 ? 0.5 : -0.5) * col.gy;
            for (int j = 0; j < Q; ++j) {
              const double num = mean ? kexact[q * Q + j] + sg * hsum(mc) : kexact[q * Q + j] - sg * col.rho_ref;
              const double d = num / (1.0 + sg);
              // dr holds the FP32 value of the same closure: what it misses of d
              const double have = hsum_node(dr[q], j);
              set_node(dl[q], j, d - have);
            }
          }
        }
      }
    };
    if (zh) {
      if (SHARED_K) __syncthreads();  // k
      if (mean) {
        sync();  // mass_s of the column before
        put_mass(mass_of<S>(mass0));
        sync();
        zmean = mean_of_mass();
      }
      closure(Kq, zmean, low_first, kx);
    }
    auto moments_mass = [&] {
      S s{};
#pragma unroll
      for (int q = 0; q < R; ++q)
        if (live(q)) s = s + item_mass(dr[q]);
      put_mass(s);
    };
    sync();  // halo zeros; mass_s free again
    if (mean) moments_mass();

    int flag = 0;
    double res = a.resid ? a.resid[c] : 0.0, best = INFINITY;
    int stalled = 0;
    const bool mpe = ACC && run.mpe_checks > 0 && run.snap != nullptr;
    int nsnap = 0, checks_since = 0;
    bool verify = false, skip_cycle = false;
    double res_before = 0.0;
    auto slot = [&](int j) { return static_cast<T*>(run.snap) + size_t(j) * size_t(run.slot) + 9 * col.node_off; };
    auto node = [&](int q) { return size_t(y0 + (item(q) >> a.row_log2)) * nx + size_t(l * Q); };

    long long it = 0;
    const long long iters = run.max_steps;
    bool last = false;
    int until = K >= 2 ? K : 0;  // steps to the end of the check interval, this one included (0: no checks)
    while (it < iters) {
      last = it + 1 == iters;
      const bool save = until == 2, chk = until == 1;
      const bool low_next = LOW && (until == 3 || until == 2 || (until == 1 && K == 2));
      if (until) until = until == 1 ? K : until - 1;
      if (save) {
#pragma unroll
        for (int q = 0; q < R; ++q)
          if (live(q)) {
            store_item(prev + node(q), dr[q]);
            if (LOW) store_item(prev + NN + node(q), dl[q]);
          }
      }
      if (chk) {  // max |rho_t - rho_(t-1)| over the column
        M rm{};
#pragma unroll
        for (int q = 0; q < R; ++q)
          if (live(q)) {
            const L pl = LOW ? load_item(prev + NN + node(q)) : zeroL;
            rm = larger(rm, item_change(dr[q], dl[q], load_item(prev + node(q)), pl));
          }
#pragma unroll
        for (int mm = 16; mm; mm >>= 1) rm = larger(rm, lane_value(rm, lane ^ mm));
        if (lane < cs) {
          M* dst = &max_s[rank * NW + warp];
          *(cs > 1 ? cluster.map_shared_rank(dst, lane) : dst) = rm;
        }
        sync();
        M rmax{};
        for (int q = 0; q < cs * NW; ++q) rmax = larger(rmax, max_s[q]);
        const double r = hsum(rmax);
        res = r;
        bool stop = false;
        if (!(r > run.tol)) {  // converged (uniform)
          last = stop = true;
        } else if (r < 0.99 * best) {
          best = r;
          stalled = 0;
        } else if (run.stall_checks > 0 && r < kStallBelow<T> && ++stalled >= run.stall_checks) {
          last = stop = true;  // no gain near the precision's rounding floor
        }
        if (ACC && mpe && !stop) {
          // ---- minimal polynomial extrapolation on the moments (see lbm_batch.cu), ahead of their
          // collision, so that a run's last step takes part too: its populations are the collision of
          // the estimate
          auto keep = [&](T* dst) {
#pragma unroll
            for (int q = 0; q < R; ++q)
              if (live(q)) {
                store_item(dst + node(q), dr[q]);
                store_item(dst + NN + node(q), jx[q]);
                store_item(dst + 2 * NN + node(q), jy[q]);
              }
          };
          auto take = [&](const T* src) {
#pragma unroll
            for (int q = 0; q < R; ++q)
              if (live(q)) {
                dr[q] = load_item(src + node(q));
                jx[q] = load_item(src + NN + node(q));
                jy[q] = load_item(src + 2 * NN + node(q));
                dl[q] = zeroL;
              }
          };
          auto remass = [&] {
            if (mean) {
              sync();
              moments_mass();
            }
          };
          if (verify) {
            // the first check after an extrapolation: a larger change than before it means the
            // estimate is worse - back to the last snapshot
            verify = false;
            if (res > res_before) {
              take(slot(kMpeK + 1));
              remass();
              skip_cycle = true;
              nsnap = 0;
              checks_since = 0;
            }
          }
          if (++checks_since >= run.mpe_checks) {
            checks_since = 0;
            keep(slot(nsnap));
            if (++nsnap == kMpeK + 2) {
              nsnap = 0;
              if (skip_cycle) {
                skip_cycle = false;
              } else {
                double G[NG];
#pragma unroll
                for (int i = 0; i < NG; ++i) G[i] = 0.0;
#pragma unroll
                for (int q = 0; q < R; ++q) {
                  if (!live(q)) continue;
                  for (int e = 0; e < 3 * Q; ++e) {  // component e / Q, node e % Q
                    const size_t at = size_t(e / Q) * NN + node(q) + size_t(e % Q);
                    double x[NU + 1];
#pragma unroll
                    for (int j = 0; j <= NU; ++j) x[j] = hsum(slot(j)[at]);
                    int p = 0;
#pragma unroll
                    for (int i = 0; i < NU; ++i)
#pragma unroll
                      for (int j = i; j < NU; ++j) G[p++] += (x[i + 1] - x[i]) * (x[j + 1] - x[j]);
                  }
                }
#pragma unroll
                for (int i = 0; i < NG; ++i) {
                  const double v = lanes_total(G[i], 32);
                  if (lane == 0) *(cs > 1 ? cluster.map_shared_rank(&gram_s[i][rank * NW + warp], 0) : &gram_s[i][warp]) = v;
                }
                sync();
                if (rank == 0 && tid == 0) {
                  double g[NG], gam[NU];
                  for (int i = 0; i < NG; ++i) {
                    g[i] = 0.0;
                    for (int w = 0; w < cs * NW; ++w) g[i] += gram_s[i][w];
                  }
                  const bool ok = mpe_solve(g, gam);
                  for (int r = 0; r < cs; ++r) {
                    double* dst = cs > 1 ? cluster.map_shared_rank(gam_s, r) : gam_s;
                    for (int j = 0; j < NU; ++j) dst[j] = gam[j];
                    *(cs > 1 ? cluster.map_shared_rank(&ok_s, r) : &ok_s) = ok ? 1 : 0;
                  }
                }
                sync();
                if (ok_s) {
                  double gam[NU];
                  for (int j = 0; j < NU; ++j) gam[j] = gam_s[j];
                  int bad = 0;
#pragma unroll
                  for (int q = 0; q < R; ++q) {
                    if (!live(q)) continue;
                    for (int e = 0; e < 3 * Q; ++e) {
                      const size_t at = size_t(e / Q) * NN + node(q) + size_t(e % Q);
                      double acc = 0.0;
                      for (int j = 0; j < NU; ++j) acc += gam[j] * hsum(slot(j)[at]);
                      if (e < Q) {
                        if (!(col.rho_ref + acc > 0.0)) bad = 1;
                        set_node(dr[q], e, acc);
                      } else if (e < 2 * Q) {
                        set_node(jx[q], e - Q, acc);
                      } else {
                        set_node(jy[q], e - 2 * Q, acc);
                      }
                    }
                    dl[q] = zeroL;
                  }
                  bad = __syncthreads_or(bad);
                  if (cs > 1) {
                    if (tid < cs) *cluster.map_shared_rank(&bad_s[rank], tid) = bad;
                    sync();
                    for (int r = 0; r < cs; ++r) bad |= bad_s[r];
                  }
                  if (bad)
                    take(slot(kMpeK + 1));  // the state before
                  remass();
                  if (!bad) {
                    verify = true;
                    res_before = res;
                  }
                }
              }
            }
          }
        }
      }
      // ---- psi and its stencil sums
      L psi[R];
#pragma unroll
      for (int q = 0; q < R; ++q) {
        if (!warp_live(q)) continue;
        const int i = item(q), s = i + P;
#pragma unroll
        for (int j = 0; j < N; ++j) {
          int fl = 0;  // lanes without a node evaluate some positive density
          const V rho = live(q) ? k.p.rho_ref + dr[q].v[j] : cst<V>(0.05);
          psi[q].v[j] = unit_psi(rho, k.k1, k.p.RT, k, fl);
          if (live(q)) flag |= fl;
        }
        const L w = left(psi[q]), e = right(psi[q]);
        L A = e - w, B;
#pragma unroll
        for (int j = 0; j < N; ++j) {
          B.v[j] = fma2(0.25, e.v[j] + w.v[j], psi[q].v[j]);
          if constexpr (kPsi2<V> == 3.0) {
            A.v[j] = scale2(0.25, A.v[j]);
          } else {
            A.v[j] = cst<V>(1.0 / 12.0) * A.v[j];
            B.v[j] = cst<V>(1.0 / 3.0) * B.v[j];
          }
        }
        if (live(q)) {
          sA[s] = A;
          sB[s] = B;
          const int r = i >> a.row_log2;
          if (cs > 1) {
            if (r == 0 && rank > 0) {
              remote(sA, rank - 1)[(rows_dn + 1) * P + l] = A;
              remote(sB, rank - 1)[(rows_dn + 1) * P + l] = B;
            }
            if (r == rows - 1 && rank < cs - 1) {
              remote(sA, rank + 1)[l] = A;
              remote(sB, rank + 1)[l] = B;
            }
          }
        }
      }
      sync();
      S mc{};  // <rho> - rho_ref of the moments
      if (mean) mc = mean_of_mass();
      const V off = mean ? zero - mean_value<V>(zh ? zmean : mc) : k.p.rho_ref;
      // ---- collision, and what each node sends
#pragma unroll
      for (int q = 0; q < R; ++q) {
        if (!warp_live(q)) continue;
        const int i = item(q), s = i + P, r = i >> a.row_log2, y = y0 + r;
        L Sx = zeroL, Sy = zeroL;
        if (live(q) && y > 0 && y < ny - 1) {
          const L A = sA[s], An = sA[s + P] + sA[s - P];
#pragma unroll
          for (int j = 0; j < N; ++j) Sx.v[j] = fma2(4.0, A.v[j], An.v[j]);
          Sy = sB[s + P] - sB[s - P];
        }
        L o[9];
#pragma unroll
        for (int j = 0; j < N; ++j) {
          V ov[9];
          unit_collide<0>(dr[q].v[j], jx[q].v[j], jy[q].v[j], psi[q].v[j], Sx.v[j], Sy.v[j], off, k, ov);
#pragma unroll
          for (int p = 0; p < 9; ++p) o[p].v[j] = ov[p];
        }
        if (last) {
          if (live(q)) {
            T* dst = f + node(q);
#pragma unroll
            for (int p = 0; p < 9; ++p) store_item(dst + p * NN, o[p]);
          }
          continue;
        }
        const L f1 = left(o[1]), f5 = left(o[5]), f8 = left(o[8]);
        const L f3 = right(o[3]), f6 = right(o[6]), f7 = right(o[7]);
        const L us = f5 + f6, vs = f8 + f7, ws = f1 + f3;
        const L u1 = o[2] + us, u2 = f5 - f6, v1 = o[4] + vs, v2 = f8 - f7;
        dr[q] = o[0] + ws;
        jx[q] = f1 - f3;
        jy[q] = zeroL;
        if (LOW && low_next) {
          const L ul = two_sum_error(f5, f6, us) + two_sum_error(o[2], us, u1);
          const L vl = two_sum_error(f8, f7, vs) + two_sum_error(o[4], vs, v1);
          dl[q] = two_sum_error(f1, f3, ws) + two_sum_error(o[0], ws, dr[q]);
          if (live(q)) {
            sul[s] = ul;
            svl[s] = vl;
            if (cs > 1 && r == rows - 1 && rank < cs - 1) remote(sul, rank + 1)[l] = ul;
            if (cs > 1 && r == 0 && rank > 0) remote(svl, rank - 1)[(rows_dn + 1) * P + l] = vl;
          }
        }
        if (!zh) {  // halfway bounce-back: no x shift (Zou-He: the closure replaces it)
          if (y == 0) {
            const L b = o[7] + o[8], n = o[4] + b;
            if (LOW && low_next)
              dl[q] = dl[q] + (two_sum_error(o[7], o[8], b) + two_sum_error(o[4], b, n) +
                               two_sum_error(dr[q], n, dr[q] + n));
            dr[q] = dr[q] + n;
            jx[q] = jx[q] + (o[7] - o[8]);
            jy[q] = n;
          }
          if (y == ny - 1) {
            const L b = o[5] + o[6], n = o[2] + b;
            if (LOW && low_next)
              dl[q] = dl[q] + (two_sum_error(o[5], o[6], b) + two_sum_error(o[2], b, n) +
                               two_sum_error(dr[q], n, dr[q] + n));
            dr[q] = dr[q] + n;
            jx[q] = jx[q] + (o[6] - o[5]);
            jy[q] = jy[q] - n;
          }
        }
        if (live(q)) {
          su1[s] = u1;
          su2[s] = u2;
          sv1[s] = v1;
          sv2[s] = v2;
          if (cs > 1) {
            if (r == rows - 1 && rank < cs - 1) {
              remote(su1, rank + 1)[l] = u1;
              remote(su2, rank + 1)[l] = u2;
            }
            if (r == 0 && rank > 0) {
              remote(sv1, rank - 1)[(rows_dn + 1) * P + l] = v1;
              remote(sv2, rank - 1)[(rows_dn + 1) * P + l] = v2;
            }
          }
        }
      }
      ++it;
      if (last) break;
      sync();
      // ---- the moments of the streamed populations
#pragma unroll
      for (int q = 0; q < R; ++q) {
        if (!live(q)) continue;
        const int s = item(q) + P;
        const L up = su1[s - P], dn = sv1[s + P], t = up + dn, d2 = dr[q] + t;
        jx[q] = jx[q] + (su2[s - P] + sv2[s + P]);
        jy[q] = jy[q] + (up - dn);
        if (LOW && low_next)
          dl[q] = dl[q] + (sul[s - P] + svl[s + P]) + (two_sum_error(up, dn, t) + two_sum_error(dr[q], t, d2));
        dr[q] = d2;
      }
      if (zh) {
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const int y = y0 + (item(q) >> a.row_log2);
          Kq[q] = y == 0 ? dr[q] - jy[q] : dr[q] + jy[q];
          if (LOW && low_next)
            for (int j = 0; j < Q; ++j)
              kx[q * Q + j] = hsum_node(dr[q], j) + hsum_node(dl[q], j) +
                              (y == 0 ? -hsum_node(jy[q], j) : hsum_node(jy[q], j));
        }
        closure(Kq, mc, low_next, kx);
        zmean = mc;
      }
      if (mean) moments_mass();
    }
    const int any = __syncthreads_or(flag);
    if (tid == 0 && any) {
      if (a.status)
        atomicOr(a.status, STATUS_NONPHYS);
      else
        atomicOr(a.col_status + c, STATUS_NONPHYS);
    }
    if (rank == 0 && tid == 0 && a.steps) {
      a.steps[c] += it;
      a.resid[c] = res;
      long long t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      a.col_ns[c] += t - t_start;
    }
  }
  sync();  // no CTA leaves while another may still write to its shared memory
}

}  // namespace
}  // namespace lbm
