// The fused D2Q9 step on moments (all relaxation times 1; arXiv 2301.12869, Sec. III, with
// Lambda = I as in Sec. IV). The physics and why three numbers a node suffice: lbm_unit.cuh.
//
// State: M_t = (drho, j_x, j_y) of the streamed populations at time t, three planes [ny][nx].
// One launch maps M_t to M_(t+1): collide, then stream (pull) - the population step's order
// started half a step earlier. The populations after t steps are f*_t = collide(M_(t-1)), and
// the state before the last step stays in the other buffer, so lbm_get_state writes them from
// there (WALK_POPULATIONS).
//
// Bound: 24 B a node and step against the population kernel's 72 B, and 87 operations a node
// (packed in pairs for FP32) against 146. FP32 is bound by a row's dependency chain with 16
// warps on an SM, FP64 by the FP64 pipe (an instruction per SM every 15.4 clocks). Measured
// against the population step, steps alone: 1024 x 4096 FP32 with <rho> 53.1 -> 22.6 us a step (4.5
// TB/s of its own 24 B), 772 x 1003 16.6 -> 6.2, 512 x 512 10.5 -> 4.3; 1024 x 4096 FP64 with <rho>
// 1293 -> 819 us (971 on populations since they collide from three moments).
//
// Layout: a warp (or a segment of 8 or 16 lanes on narrow lattices) walks a strip of rows
// upward. A lane holds two columns of a row, an FP32 pair or two FP64 values (two FP32 pairs a
// lane need 168 registers and leave 12 warps an SM: 23.7 us); the first and last lane
// of a segment are halo (x periodic: a lane's columns are taken modulo nx, which its width
// divides). x neighbours come from the adjacent lane by one shuffle a quantity, y neighbours
// from a three-row window in registers, so there is no shared memory and no barrier in the
// walk. At input row q: psi of row q; collision of row q - 1; row q - 2 receives its last
// contributions and is stored. Of the nine post-collision values the walk keeps column sums
// only: for target row y
//   V = f0(y) + f2(y-1) + f4(y+1)                                     (from x)
//   P = f1(y) + f5(y-1) + f8(y+1),  D = f5(y-1) - f8(y+1)             (from x - 1)
//   Q = f3(y) + f6(y-1) + f7(y+1),  E = f6(y-1) - f7(y+1)             (from x + 1)
// so drho = V + P + Q, j_x = P - Q, j_y = f2(y-1) - f4(y+1) + D + E: four shuffled values
// instead of six. The row loop runs three rows an iteration so that the windows rotate by
// register renaming; rows are loaded three ahead.
#include "lbm_dd.cuh"
#include "lbm_internal.h"
#include "lbm_lane.cuh"
#include "lbm_ptx.cuh"
#include "lbm_unit.cuh"

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace lbm {
namespace {

// ---- the columns of a row that a lane holds: N values (FP32 pairs, or FP64 columns)
template <typename T>
struct LaneOf;
template <>
struct LaneOf<float> {
  using V = f2;
  static constexpr int N = 1;
};
template <>
struct LaneOf<double> {
  using V = double;
  static constexpr int N = 2;
};
template <typename T>
using LaneT = Lane<typename LaneOf<T>::V, LaneOf<T>::N>;
template <typename T>
constexpr int kColumns = LaneOf<T>::N* VecTraits<typename LaneOf<T>::V>::width;  // a lane's columns

__device__ __forceinline__ Lane<f2, 1> load_lane(const float* p) {
  return {{*reinterpret_cast<const f2*>(p)}};
}
__device__ __forceinline__ Lane<double, 2> load_lane(const double* p) {
  const double2 q = *reinterpret_cast<const double2*>(p);
  return {{q.x, q.y}};
}
__device__ __forceinline__ void store_lane(float* p, const Lane<f2, 1>& q) {
  *reinterpret_cast<f2*>(p) = q.v[0];
}
__device__ __forceinline__ void store_lane(double* p, const Lane<double, 2>& q) {
  *reinterpret_cast<double2*>(p) = make_double2(q.v[0], q.v[1]);
}
// into a caller's array of doubles, which may start on any 8-byte boundary
__device__ __forceinline__ void store_doubles(double* p, const Lane<double, 2>& q) {
  if (reinterpret_cast<uintptr_t>(p) & 15u) {
    p[0] = q.v[0];
    p[1] = q.v[1];
  } else {
    store_lane(p, q);
  }
}
template <int N>
__device__ __forceinline__ void store_doubles(double* p, const Lane<f2, N>& q) {
#pragma unroll
  for (int j = 0; j < N; ++j) store_doubles(p + 2 * j, Lane<double, 2>{{lo(q.v[j]), hi(q.v[j])}});
}

// value at x - 1 / x + 1 of every column; the segment's edge lanes get their own value there
template <typename V, int N>
__device__ __forceinline__ Lane<V, N> from_left(const Lane<V, N>& q, int seg) {
  return shift_left(q, [seg](auto v) { return __shfl_up_sync(0xffffffffu, v, 1, seg); });
}
template <typename V, int N>
__device__ __forceinline__ Lane<V, N> from_right(const Lane<V, N>& q, int seg) {
  return shift_right(q, [seg](auto v) { return __shfl_down_sync(0xffffffffu, v, 1, seg); });
}

// sum over the warp of the lanes' mass partials, in every lane: the FP32 accumulators' two-sum
// pairs are added as pairs (48 bits), since FP64 conversions and additions issue at 1/64 of
// the FP32 rate
__device__ __forceinline__ double warp_total(double s) { return warp_sum(s); }
__device__ __forceinline__ dd warp_total(dd s) {
#pragma unroll
  for (int m = 16; m; m >>= 1)
    s = s + dd{__shfl_xor_sync(0xffffffffu, s.hi, m), __shfl_xor_sync(0xffffffffu, s.lo, m)};
  return s;
}
__device__ __forceinline__ double lane_mass(const Acc<double>& a) { return a.value(); }
__device__ __forceinline__ dd lane_mass(const Acc<f2>& a) {
  return dd{lo(a.hi[0]), lo(a.lo[0])} + dd{hi(a.hi[0]), hi(a.lo[0])};
}
// the CTA's total into out[blockIdx.x]; red: one value a warp
template <typename V, typename S>
__device__ __forceinline__ void cta_mass(const Acc<V>& acc, S* red, double* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const S v = warp_total(lane_mass(acc));
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    const S t = warp_total(lane < int(blockDim.x >> 5) ? red[lane] : S{});
    if (lane == 0) out[blockIdx.x] = hsum(t);
  }
}
template <typename V>
using MassOf = decltype(lane_mass(Acc<V>{}));

template <typename T, int MODE, bool TH, bool MEAN>
__global__ void __launch_bounds__(sizeof(T) == 4 ? kWalkThreadsF : kWalkThreadsD, 1)
    walk_kernel(const WalkTiling tl, const UnitT<typename LaneOf<T>::V> k, const WalkIO io) {
  using V = typename LaneOf<T>::V;
  using L = LaneT<T>;
  constexpr int N = LaneOf<T>::N, W = kColumns<T>;
  constexpr int HALO = MODE == WALK_STEP ? 2 : 1;  // rows read beyond the strip on each side
  __shared__ double mean_s[2];
  __shared__ MassOf<V> sums[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nx = tl.nx, ny = tl.ny, seg = tl.seg;
  // this segment's band and strip; segments past the last strip own nothing (they stay with
  // their warp for its shuffles)
  const int item = (blockIdx.x * blockDim.x + tid) / seg;
  const int l = tid & (seg - 1);
  const int band = item % tl.nbands, strip = item / tl.nbands;
  const int ya = strip * tl.strip_h, yb = min(ya + tl.strip_h, ny);
  const int c0 = band * tl.band_w + (l - 1) * W;  // first column, unwrapped
  const bool own = l >= 1 && l < seg - 1 && c0 < min(band * tl.band_w + tl.band_w, nx);
  int x = c0 % nx;
  if (x < 0) x += nx;
  const size_t plane = size_t(nx) * ny;
  const T* mdr = static_cast<const T*>(io.min) + x;
  const T* Tf = TH ? static_cast<const T*>(io.Tfield) + x : nullptr;
  const bool zh = tl.zh != 0;
  griddep_wait();  // launched as a dependent of the previous kernel: its state is complete
  griddep_launch_dependents();
  if (MODE == WALK_POPULATIONS && io.pending && *io.pending == 0) return;

  struct Raw {
    L dr, jx, jy, t;
  };
  // rows beyond the strip's reach or the lattice load the nearest one that is not: what is
  // formed from them is never used
  const int q_top = min(yb + HALO, ny) - 1;
  auto fetch = [&](int q, Raw& w) {
    const size_t n = size_t(max(min(q, q_top), 0)) * nx;
    w.dr = load_lane(mdr + n);
    w.jx = load_lane(mdr + plane + n);
    w.jy = load_lane(mdr + 2 * plane + n);
    if constexpr (TH) w.t = load_lane(Tf + n);
  };
  const int q0 = ya - HALO;
  Raw r0, r1, r2;
  fetch(q0, r0);
  fetch(q0 + 1, r1);
  fetch(q0 + 2, r2);

  // <rho> - rho_ref for the collision, and with Zou-He walls the one of the closure (the mass
  // of the populations about to be streamed = the sum of drho now, since the collision keeps
  // it). Warp 0 sums and announces it (bar.arrive) while the others form psi of their first rows,
  // and goes on to its own: nobody waits for warp 0's psi. Then only psi of the first two rows is
  // formed ahead of it, their collision is not needed (without <rho> there is nothing to wait for, and
  // leaving those collisions out was slower). Whole passes - a state set, a block of steps, the state and
  // rho read - over their steps: 256 x 768 (200 steps) 6.38 -> 6.25 us, 1024 x 4096 FP64 (10) 1018 -> 1007;
  // 772 x 1003 without <rho> (150) 7.18, without those collisions 7.29.
  const V zero = cst<V>(0.0);
  const L zero2 = splat_lane<V, N>(zero);
  V dmean = zero, dclose = zero;
  auto take_mean = [&] {
    dclose = cst<V>(mean_s[0]);
    dmean = cst<V>(mean_s[1]);
  };
  if (MEAN && warp == 0) {
    const double s = warp_sum_partials(io.part_in, io.npart_in);
    if (lane == 0) {
      const double m = s * tl.inv_n_total;
      mean_s[0] = m;
      mean_s[1] = zh ? *io.mean_in : m;
      if (MODE == WALK_STEP && zh && blockIdx.x == 0) *io.mean_out = m;
    }
    __syncwarp();
    take_mean();
    asm volatile("bar.arrive 1, %0;" ::"r"(blockDim.x) : "memory");
  }
  auto wait_mean = [&] {
    if (MEAN && warp != 0) {
      asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x) : "memory");
      take_mean();
    }
  };

  int flag = 0;
  Acc<V> acc;
  // psi of row q - 1; (1/12) d of row q - 1, (1/3) d(q - 1) + (1/12) d(q - 2), and
  // (1/3) psi + (1/12) s of rows q - 2, q - 1 (d, s: psi(x+1) -+ psi(x-1))
  L psi1 = zero2, A1 = zero2, X1 = zero2, B0 = zero2, B1 = zero2;
  L dr1 = zero2, jx1 = zero2, jy1 = zero2;  // moments of row q - 1
  L V1 = zero2, P1 = zero2, Q1 = zero2;     // f2, f5, f6 of row q - 2 (for target q - 1)
  // target q - 2 so far: sums from rows q-3 and q-2, its southern f2, f5, f6, and what the
  // bottom wall sends back without an x shift
  L S2 = zero2, P2 = zero2, Q2 = zero2, a2 = zero2, a5 = zero2, a6 = zero2, Jh = zero2;
  const V c13 = cst<V>(1.0 / 3.0), c112 = cst<V>(1.0 / 12.0);

  // EDGE: rows at the walls or beyond may take part; COLL: row q - 1 collides (the first two rows
  // of a strip only start the windows)
  auto body = [&](int q, Raw& in, auto edge, auto coll) {
    constexpr bool EDGE = decltype(edge)::value, COLL = decltype(coll)::value;
    // ---- psi of row q
    const L dr2 = in.dr, jx2 = in.jx, jy2 = in.jy;
    L psi2;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      if constexpr (TH)
        psi2.v[j] = unit_psi(k.p.rho_ref + dr2.v[j], k.k1R * in.t.v[j], k.p.R * in.t.v[j], k, flag);
      else
        psi2.v[j] = unit_psi(k.p.rho_ref + dr2.v[j], k.k1, k.p.RT, k, flag);
    }
    fetch(q + 3, in);
    const L w = from_left(psi2, seg), e = from_right(psi2, seg);
    const L d2 = e - w;
    const L A2 = c112 * d2;
    const L B2 = fma_lane(c13, psi2, c112 * (e + w));
    // ---- collision of row r = q - 1 (Eq. ShanChenForce stencil; zero on the wall rows)
    const int r = q - 1;
    L Sx = X1 + A2, Sy = B2 - B0;
    if (EDGE && (r <= 0 || r >= ny - 1)) Sx = Sy = zero2;
    X1 = fma_lane(c13, d2, A1);
    A1 = A2;
    B0 = B1;
    B1 = B2;
    L rho, ux, uy;
    if constexpr (!COLL) {
    } else if constexpr (MODE == WALK_MOMENTS) {
#pragma unroll
      for (int j = 0; j < N; ++j) {
        V Fx, Fy;
        const Velocity<V> u =
            unit_velocity<MEAN ? 2 : 1>(dr1.v[j], jx1.v[j], jy1.v[j], psi1.v[j], Sx.v[j], Sy.v[j], dmean, k, Fx, Fy);
        rho.v[j] = u.rho;
        ux.v[j] = u.ux;
        uy.v[j] = u.uy;
      }
      if (own && r >= ya && r < yb) {
        const size_t n = size_t(r) * nx + x;
        if (io.rho_out) store_doubles(io.rho_out + n, rho);
        if (io.ux_out) store_doubles(io.ux_out + n, ux);
        if (io.uy_out) store_doubles(io.uy_out + n, uy);
      }
    } else {
      L f[9];
#pragma unroll
      for (int j = 0; j < N; ++j) {
        V o[9];
        const Velocity<V> u =
            unit_collide<MEAN ? 2 : 1>(dr1.v[j], jx1.v[j], jy1.v[j], psi1.v[j], Sx.v[j], Sy.v[j], dmean, k, o);
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i].v[j] = o[i];
        rho.v[j] = u.rho;
        ux.v[j] = u.ux;
        uy.v[j] = u.uy;
      }
      if constexpr (MODE == WALK_POPULATIONS) {
        if (own && r >= ya && r < yb) {
          T* dst = static_cast<T*>(io.fout) + size_t(r) * nx + x;
#pragma unroll
          for (int i = 0; i < 9; ++i) store_lane(dst + i * plane, f[i]);
        }
      } else {
        if (TH && own && r >= ya && r < yb) {  // this step's rho, u for the energy equation
          const size_t n = size_t(r) * nx + x;
          store_lane(static_cast<T*>(io.rho_T) + n, rho);
          store_lane(static_cast<T*>(io.ux_T) + n, ux);
          store_lane(static_cast<T*>(io.uy_T) + n, uy);
        }
        // ---- target y = q - 2 receives row r's f4, f8, f7; past the top wall row (r = ny) row
        // ny - 1's own f2, f5, f6 come back instead (halfway bounce-back)
        const int y = r - 1;
        L n4 = f[4], n8 = f[8], n7 = f[7];
        if (EDGE && r == ny) {
          n4 = n8 = n7 = zero2;
          if (!zh) {
            n4 = V1 + (P1 + Q1);
            Jh = Jh + (Q1 - P1);
          }
        }
        const L Ps = from_left(P2 + n8, seg), Ds = from_left(a5 - n8, seg);
        const L Qs = from_right(Q2 + n7, seg), Es = from_right(a6 - n7, seg);
        L dr = (S2 + n4) + (Ps + Qs);
        L jx = Ps - Qs;
        L jy = (a2 - n4) + (Ds + Es);
        if (EDGE && (y == 0 || y == ny - 1)) {
          jx = jx + Jh;
          if (zh) {
            const L K = y == 0 ? dr - jy : dr + jy;
#pragma unroll
            for (int j = 0; j < N; ++j) unit_zou_he(K.v[j], y == 0, dclose, k, dr.v[j], jx.v[j], jy.v[j]);
          }
        }
        if (own && y >= ya && y < yb) {
          T* dst = static_cast<T*>(io.mout) + size_t(y) * nx + x;
          store_lane(dst, dr);
          store_lane(dst + plane, jx);
          store_lane(dst + 2 * plane, jy);
          if (MEAN) acc.add(sum_lane(dr));
        }
        // ---- target r: its own f0, f1, f3 on top of row r - 1's f2, f5, f6; at the bottom wall
        // its f4, f7, f8 come back (Zou-He: the closure replaces them)
        a2 = V1;
        a5 = P1;
        a6 = Q1;
        if (EDGE) Jh = zero2;
        if (EDGE && r == 0) {
          a2 = a5 = a6 = zero2;
          if (!zh) {
            a2 = f[4] + (f[7] + f[8]);
            Jh = f[7] - f[8];
          }
        }
        S2 = a2 + f[0];
        P2 = a5 + f[1];
        Q2 = a6 + f[3];
        V1 = f[2];
        P1 = f[5];
        Q1 = f[6];
      }
    }
    dr1 = dr2;
    jx1 = jx2;
    jy1 = jy2;
    psi1 = psi2;
  };
  // input rows ya - HALO .. yb + HALO - 1 (a step stores row yb - 1 at q = yb + 1), three at a
  // time; away from the walls without their cases (uniform over the warp)
  const int nq = tl.strip_h + 2 * HALO;
  const std::true_type yes{};
  const std::false_type no{};
  body(q0, r0, yes, std::bool_constant<!MEAN>{});
  body(q0 + 1, r1, yes, std::bool_constant<!MEAN>{});
  wait_mean();
  body(q0 + 2, r2, yes, yes);
  for (int it = 3; it < nq; it += 3) {
    const int q = q0 + it;
    if (MODE == WALK_STEP && __all_sync(0xffffffffu, q >= 3 && q + 2 < ny)) {
      body(q, r0, no, yes);
      body(q + 1, r1, no, yes);
      body(q + 2, r2, no, yes);
    } else {
      body(q, r0, yes, yes);
      body(q + 1, r1, yes, yes);
      body(q + 2, r2, yes, yes);
    }
  }

  const int wf = __reduce_or_sync(0xffffffffu, flag);
  if (lane == 0 && wf) atomicOr(io.status, wf);
  if (MODE == WALK_STEP && MEAN) {
    cta_mass(acc, sums, io.part_out);
  }
}

// a lane's columns of a row at x, each with its neighbour at x - 1 (LEFT) or x + 1 instead;
// xn: the neighbour beyond the lane's columns
template <bool LEFT>
__device__ __forceinline__ Lane<f2, 1> shift(const float* p, int x, int xn, std::bool_constant<LEFT>) {
  const Lane<f2, 1> c = load_lane(p + x);
  if (LEFT) return {{make_f2(p[xn], lo(c.v[0]))}};
  return {{make_f2(hi(c.v[0]), p[xn])}};
}
template <bool LEFT>
__device__ __forceinline__ Lane<double, 2> shift(const double* p, int x, int xn, std::bool_constant<LEFT>) {
  const Lane<double, 2> c = load_lane(p + x);
  if (LEFT) return {{p[xn], c.v[0]}};
  return {{c.v[1], p[xn]}};
}

// ---- populations -> moments: M_t of the stored f*_t (Eqs. LBE, Density, Momentum without the
// force), and its FP64 partial sums, as many as a walk's; one thread a lane's columns of a row. The
// loads want all the warps an SM takes: 1024 x 4096, cold: FP32 111 us with 8 warps a CTA, 39 with 32;
// FP64 202, 150 with 16 (the FP64 pipe's)
template <typename T>
constexpr int kPullThreads = sizeof(T) == 4 ? 1024 : 512;
template <typename T>
__global__ void __launch_bounds__(kPullThreads<T>, 1) pull_kernel(const WalkTiling tl, const UnitT<typename LaneOf<T>::V> k,
                                                   const WalkIO io) {
  using V = typename LaneOf<T>::V;
  using L = LaneT<T>;
  constexpr int N = LaneOf<T>::N, W = kColumns<T>;
  __shared__ double mean_s;
  __shared__ MassOf<V> sums[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nx = tl.nx, ny = tl.ny, groups = nx / W;
  const size_t plane = size_t(nx) * ny;
  const T* f = static_cast<const T*>(io.fin);
  const bool zh = tl.zh != 0;
  V dclose = cst<V>(0.0);
  if (k.p.form == 2 && zh) {  // <rho> of the closure: the stored populations' mass
    if (warp == 0) {
      const double s = warp_sum_partials(io.part_in, io.npart_in);
      if (lane == 0) {
        mean_s = s * tl.inv_n_total;
        if (blockIdx.x == 0) *io.mean_out = mean_s;
      }
    }
    __syncthreads();
    dclose = cst<V>(mean_s);
  }
  Acc<V> acc;
  const size_t total = size_t(groups) * ny;
  for (size_t g = blockIdx.x * size_t(blockDim.x) + tid; g < total; g += size_t(gridDim.x) * blockDim.x) {
    const int y = int(g / groups), x = int(g - size_t(y) * groups) * W;
    const int xl = x == 0 ? nx - 1 : x - 1, xr = x + W == nx ? 0 : x + W;
    auto at = [&](int i, int row) { return f + i * plane + size_t(row) * nx; };
    auto centre = [&](int i, int row) { return load_lane(at(i, row) + x); };
    auto west = [&](int i, int row) { return shift(at(i, row), x, xl, std::true_type{}); };
    auto east = [&](int i, int row) { return shift(at(i, row), x, xr, std::false_type{}); };
    const bool lo_w = y == 0, hi_w = y == ny - 1;
    const L f0 = centre(0, y), f1 = west(1, y), f3 = east(3, y);
    const L f2_ = lo_w ? centre(4, y) : centre(2, y - 1);
    const L f5 = lo_w ? centre(7, y) : west(5, y - 1);
    const L f6 = lo_w ? centre(8, y) : east(6, y - 1);
    const L f4 = hi_w ? centre(2, y) : centre(4, y + 1);
    const L f7 = hi_w ? centre(5, y) : east(7, y + 1);
    const L f8 = hi_w ? centre(6, y) : west(8, y + 1);
    const L P = (f1 + f5) + f8, Q = (f3 + f6) + f7;
    L dr = ((f0 + f2_) + f4) + (P + Q);
    L jx = P - Q;
    L jy = (f2_ - f4) + ((f5 - f8) + (f6 - f7));
    if (zh && (lo_w || hi_w)) {
      const L K = lo_w ? (f0 + (f1 + f3)) + cst<V>(2.0) * (f4 + (f7 + f8))
                            : (f0 + (f1 + f3)) + cst<V>(2.0) * (f2_ + (f5 + f6));
#pragma unroll
      for (int j = 0; j < N; ++j) unit_zou_he(K.v[j], lo_w, dclose, k, dr.v[j], jx.v[j], jy.v[j]);
    }
    T* dst = static_cast<T*>(io.mout) + size_t(y) * nx + x;
    store_lane(dst, dr);
    store_lane(dst + plane, jx);
    store_lane(dst + 2 * plane, jy);
    acc.add(sum_lane(dr));
  }
  if (k.p.form == 2) {
    cta_mass(acc, sums, io.part_out);
  }
}

// ---- rho alone of a state held as moments: no stencil is needed, only the test that psi^2 >= 0, the
// sign of N D without the division. FP64 densities are tested in FP32 first and again in FP64 where
// that leaves a doubt, so the slow pipe does one addition a node. 1024 x 4096, cold: 39 us by the walk
// -> 19 in FP32, 645 -> 26 in FP64
template <typename T>
struct DensityT {
  T rho_ref, b4, k1, k2, k3;  // k1: 2 RT/G, or with a temperature field 2 R/G
};
// psi^2 < 0, NaN or rho <= 0; with SURE also where rounding may decide
template <bool SURE, typename T>
__device__ __forceinline__ bool nonphysical(T rho, T b4, T k1, T k2, T k3) {
  const T eta = b4 * rho, om = T(1) - eta, D = om * om * om;
  const T A = k1 * fma(eta, fma(eta, om, T(1)), T(1)), B = fma(k2, rho, k3) * D;
  if (SURE) return !(rho > T(1e-30) && D > T(1e-3) && A + B > T(1e-5) * (fabs(A) + fabs(B)));
  return !(rho > T(0) && rho * (A + B) * D >= T(0));
}
template <typename T, bool TH>
__global__ void __launch_bounds__(256) density_kernel(const DensityT<T> k, double rho_ref, const T* __restrict__ dr,
                                                      const T* __restrict__ Tf, double* __restrict__ out, size_t n,
                                                      int* status) {
  using T2 = std::conditional_t<sizeof(T) == 4, float2, double2>;
  const float b4 = float(k.b4), k1f = float(k.k1), k2 = float(k.k2), k3 = float(k.k3);
  bool bad = false;
  auto density = [&](T d, T t) {
    const double r = widen(d) + rho_ref;
    if constexpr (sizeof(T) == 4)
      bad |= nonphysical<false>(k.rho_ref + d, b4, TH ? k1f * t : k1f, k2, k3);
    else if (nonphysical<true>(narrow(r), b4, TH ? k1f * narrow(t) : k1f, k2, k3))
      bad |= nonphysical<false>(r, k.b4, TH ? k.k1 * t : k.k1, k.k2, k.k3);
    return r;
  };
  for (size_t q = blockIdx.x * size_t(blockDim.x) + threadIdx.x; q < n / 2; q += size_t(gridDim.x) * blockDim.x) {
    const T2 d = reinterpret_cast<const T2*>(dr)[q];
    T2 t{};
    if constexpr (TH) t = reinterpret_cast<const T2*>(Tf)[q];
    out[2 * q] = density(d.x, t.x);
    out[2 * q + 1] = density(d.y, t.y);
  }
  if (bad) atomicOr(status, STATUS_NONPHYS);
}
}  // namespace

// The band layout (8, 16 or 32 lanes a segment) that wastes the fewest halo lanes, and the strip
// height with the smallest estimated time. A wave of warps takes t0 + rows x (time of a row with
// w warps on an SM): measured for FP32 0.22 us a row with 2 warps (its latency), 0.30 with 8,
// 0.50 with 16; an FP64 row is bound by the SM's FP64 pipe (1.57 us a warp: 100 issue slots of
// 15.4 clocks a column) and takes 5 us alone. 1024 x 4096 FP32: 31-row strips, one wave of
// 16 warps per SM, 22.5 us; 30 rows (two waves) 41 us, 50 rows (10 warps per SM) 27.6 us.
bool plan_walk(int precision, int nx, int ny, bool zh, int nsm, int max_ctas, WalkTiling* t) {
  const bool fp32 = precision == 1;
  const int W = fp32 ? kColumns<float> : kColumns<double>;
  t->nx = nx;
  t->ny = ny;
  t->zh = zh ? 1 : 0;
  t->inv_n_total = 1.0 / (double(nx) * double(ny));
  long best_lanes = 0;
  for (int seg : {32, 16, 8}) {
    const int own = (seg - 2) * W;
    const int nb = (nx + own - 1) / own;
    if (best_lanes == 0 || long(nb) * seg < best_lanes) {
      best_lanes = long(nb) * seg;
      t->seg = seg;
      t->nbands = nb;
    }
  }
  t->band_w = ((nx + t->nbands - 1) / t->nbands + W - 1) / W * W;
  t->nbands = (nx + t->band_w - 1) / t->band_w;
  const int most_warps = (fp32 ? kWalkThreadsF : kWalkThreadsD) / 32;
  // warps a CTA takes: a share of an SM, or more where the partial sums' slots bound the grid (1024 x 30
  // FP32 between wet walls has 60 for 180 warps in strips of 3 rows)
  auto set_rows = [&](int h) {
    t->strip_h = h;
    t->nstrips = (ny + h - 1) / h;
    const long warps = (long(t->nstrips) * t->nbands * t->seg + 31) / 32;
    const long share = (warps + nsm - 1) / nsm, slots = std::max(max_ctas, 1);
    const int per_cta = int(std::min<long>(most_warps, std::max(share, (warps + slots - 1) / slots)));
    t->threads = 32 * per_cta;
    t->ctas = int((warps + per_cta - 1) / per_cta);
    return t->ctas <= max_ctas;
  };
  double best = 0.0;
  int best_h = ny;
  for (int h = 1; h <= ny; h = h < 32 ? h + 1 : h + h / 16) {
    if (!set_rows(h)) continue;
    const double waves = double((t->ctas + nsm - 1) / nsm), w = double(t->threads / 32);
    const double row = fp32 ? 0.18 + 0.02 * w : std::max(5.0, 1.57 * w);
    const double time = waves * (1.4 + (h + 6) / 3 * 3 * row);
    if (best == 0.0 || time < best) {
      best = time;
      best_h = h;
    }
  }
  return set_rows(best_h);
}

// Estimates in us, fitted to 75 lattices of 6e4 to 4e6 nodes in both gravity forms (FP64 population step
// within 3 %, the walks within 10 %). A strip's rows, with six of halo and rounding, take a wave of the
// walk 0.18 + 0.02 w us each with w warps on an SM, in FP64 max(5.8, 0.6 + 1.45 w); a row of the population
// step 1.3 us (or the HBM's time for 72 B a node), in FP64 1.65 + 5 us a warp of 32 columns; FP64 thermal
// ones of fewer than 3e5 nodes lose some 50 us beside Heun's blocks. Forming the populations is a walk with
// nine planes to store, forming the moments a pass over memory.
StepCosts step_costs(int precision, const WalkTiling& t, int nsm, int step_band_w, int step_strip_h, int form,
                     bool thermal) {
  const double nodes = double(t.nx) * t.ny, h = step_strip_h;
  const int waves = (t.ctas + nsm - 1) / nsm, w = t.threads / 32, rows = (t.strip_h + 6) / 3 * 3;
  StepCosts c;
  if (precision == 1) {
    c.walk = waves * (1.4 + rows * (0.18 + 0.02 * w)) + (form == 2 ? 2.0 : 0.0);
    c.step = std::max(6.7 + 1.3 * h, 72.0 * nodes / 5.7e6);
    c.populations = std::max(2.0 + 0.9 * c.walk, 48.0 * nodes / 6e6);
    c.pull = 2.0 + 9e-6 * nodes;
  } else {
    const int n = (step_band_w + 31) / 32;
    c.walk = waves * (rows * std::max(5.8, 0.6 + 1.45 * w) - 4.0);
    const double r = step_strip_h == t.ny ? h - 0.8 : h;  // (the wall rows have no stencil)
    c.step = 9.3 + 1.4 * n + (1.65 + 5.0 * n) * r + (form == 2 ? 4.0 : 0.0) + (thermal && nodes < 3e5 ? 50.0 : 0.0);
    c.populations = 5.0 + 0.9 * c.walk;
    c.pull = 8.0 + 3.6e-5 * nodes;
  }
  return c;
}

// FP32 walks win everywhere (24 B a node against 72). In FP64 both steps take the FP64 pipe's time, in
// whole rows, and which is less depends on how the rows fall out: 32 x 2100 walks in 49.2 us a step and
// takes 30.9 on populations, 64 x 3000 81.8 and 58.2, 512 x 512 83.6 and 81.0, 60 x 1200 34.1 and 38.7
// (with <rho>), 1024 x 1024 227 and 255, 4 x 20000 84 and 190. Where they are alike the walk is taken:
// the density of a state on moments costs nothing like a step (100 x 3000, a step and rho: 116 us, 190
// on populations).
bool walk_pays(int precision, const WalkTiling& t, int nsm, int step_band_w, int step_strip_h, int form) {
  if (precision == 1) return true;
  const StepCosts c = step_costs(precision, t, nsm, step_band_w, step_strip_h, form, false);
  return c.walk < 1.05 * c.step;
}

namespace {
// FP64 thermal steps ask for more than half of an SM's shared memory, which they do not use, so that an
// SM takes one of their blocks. The next step's blocks start beside the last ones of Heun's kernel, and
// without that two of them (one has 3 to 8 warps) land on an SM that Heun has left while others get none:
// 1024 x 1024 628 us a step in a block of steps for walk 240 and Heun 216 alone, 448 with it; 470 x 992
// 317 and 222. Blocks of an isothermal step or an FP32 one come out the same either way.
template <typename T, int MODE, bool TH>
constexpr int kWalkShared = sizeof(T) == 8 && TH && MODE == WALK_STEP ? 120 * 1024 : 0;

template <typename T, int MODE, bool TH>
cudaError_t launch_walk_m(const WalkTiling& t, const StepPhys& ph, const WalkIO& io, cudaStream_t s) {
  const auto k = to_unit<typename LaneOf<T>::V>(ph);
  auto fn = ph.form == 2 ? walk_kernel<T, MODE, TH, true> : walk_kernel<T, MODE, TH, false>;
  return launch_dependent(fn, dim3(t.ctas), dim3(t.threads), kWalkShared<T, MODE, TH>, s, t, k, io);
}
template <typename T>
cudaError_t launch_walk_t(int mode, const WalkTiling& t, const StepPhys& ph, const WalkIO& io, cudaStream_t s) {
  const bool th = io.Tfield != nullptr;
  if (mode == WALK_STEP)
    return th ? launch_walk_m<T, WALK_STEP, true>(t, ph, io, s) : launch_walk_m<T, WALK_STEP, false>(t, ph, io, s);
  if (mode == WALK_POPULATIONS)
    return th ? launch_walk_m<T, WALK_POPULATIONS, true>(t, ph, io, s)
              : launch_walk_m<T, WALK_POPULATIONS, false>(t, ph, io, s);
  return th ? launch_walk_m<T, WALK_MOMENTS, true>(t, ph, io, s) : launch_walk_m<T, WALK_MOMENTS, false>(t, ph, io, s);
}
}  // namespace

cudaError_t walk_prepare(int precision) {
  if (precision == 1) return cudaSuccess;
  constexpr int bytes = kWalkShared<double, WALK_STEP, true>;
  const cudaError_t e = cudaFuncSetAttribute(walk_kernel<double, WALK_STEP, true, false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(walk_kernel<double, WALK_STEP, true, true>,
                                                     cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t launch_walk(int precision, int mode, const WalkTiling& t, const StepPhys& ph, const WalkIO& io,
                        cudaStream_t stream) {
  // a thermal step stores its rho, u: refuse a launch without somewhere to put them
  if (io.Tfield && mode == WALK_STEP && !(io.rho_T && io.ux_T && io.uy_T)) return cudaErrorInvalidValue;
  return precision == 1 ? launch_walk_t<float>(mode, t, ph, io, stream)
                        : launch_walk_t<double>(mode, t, ph, io, stream);
}

cudaError_t launch_pull(int precision, const WalkTiling& t, const StepPhys& ph, const WalkIO& io, cudaStream_t stream) {
  if (precision == 1)
    pull_kernel<float><<<t.ctas, kPullThreads<float>, 0, stream>>>(t, to_unit<f2>(ph), io);
  else
    pull_kernel<double><<<t.ctas, kPullThreads<double>, 0, stream>>>(t, to_unit<double>(ph), io);
  return cudaGetLastError();
}

namespace {
template <typename T>
void density(const StepPhys& ph, const void* dr, const void* Tf, double* rho, size_t n, int* status, cudaStream_t s) {
  const DensityT<T> k{T(ph.rho_ref), T(ph.b / 4.0), T(2.0 * (Tf ? ph.R : ph.RT) / ph.G), T(-2.0 * ph.a / ph.G),
                      T(-2.0 / (3.0 * ph.G))};
  const int grid = int(std::min<size_t>(4096, (n / 2 + 255) / 256));
  if (Tf)
    density_kernel<T, true><<<grid, 256, 0, s>>>(k, ph.rho_ref, static_cast<const T*>(dr), static_cast<const T*>(Tf),
                                                 rho, n, status);
  else
    density_kernel<T, false><<<grid, 256, 0, s>>>(k, ph.rho_ref, static_cast<const T*>(dr), nullptr, rho, n, status);
}
}  // namespace

cudaError_t launch_density(int precision, const StepPhys& ph, const void* dr, const void* Tfield, double* rho, size_t n,
                           int* status, cudaStream_t stream) {
  if (precision == 1)
    density<float>(ph, dr, Tfield, rho, n, status, stream);
  else
    density<double>(ph, dr, Tfield, rho, n, status, stream);
  return cudaGetLastError();
}

}  // namespace lbm
