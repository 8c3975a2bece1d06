// Per-node physics of the step when every relaxation time is 1 (Lambda = I, the paper's
// setting, Sec. IV), shared by the moment-walk kernels (lbm_walk.cu) and the batched columns
// (lbm_batch.cu).
//
// With Lambda = I, Eq. LBE's collision is m* = m_eq + S~/2 (Eqs. OperatorMRT, LiFS): the
// post-collision populations depend on the pulled ones only through rho and j. So a node's
// state can be held as three numbers - drho = rho - rho_ref, j_x, j_y of the streamed
// populations - instead of nine, and a step is: psi from rho, the Shan-Chen stencil, F and u,
// the nine post-collision values (in registers), and the three sums of the ones the
// neighbours send. The collision itself simplifies: with s = u_x g_x + u_y g_y and
// g = rho u + F, the energy moments are e* = A - 2 drho and eps* = drho - A with
// A = 3 s + (sigma/(tau - 1/2)) G^2 |S|^2 / 2, p_xx* = u_x g_x - u_y g_y,
// p_xy* = (u_x g_y + u_y g_x)/2, j* = j + F, q* = -j*. 46 operations a node instead of 78.
#pragma once

#include "lbm_dd.cuh"
#include "lbm_physics.cuh"

namespace lbm {

template <typename V>
struct UnitT {
  PhysT<V> p;
  V k1, k1R;  // 2RT/G, 2R/G
};

template <typename V>
UnitT<V> to_unit(const StepPhys& s) {
  UnitT<V> u;
  u.p = to_phys<V>(s);
  u.k1 = host_value<V>(2.0 * s.RT / s.G);
  u.k1R = host_value<V>(2.0 * s.R / s.G);
  return u;
}

// powers of two scale both parts of a double-float value exactly
__device__ __forceinline__ dd scale2(double c, dd x) { return dd{float(c) * x.hi, float(c) * x.lo}; }
__device__ __forceinline__ dd fma2(double c, dd x, dd y) { return scale2(c, x) + y; }

// ---- reciprocals of FP32 pairs and of double-float values
__device__ __forceinline__ f2 unit_rcp(f2 x) { return make_f2(rcp_approx(lo(x)), rcp_approx(hi(x))); }

// double-float: an FP32 guess (refined to 2^-23), whose correction is formed in FP32 from the
// exact remainder, so the result is good to about 2^-46
__device__ __forceinline__ dd unit_rcp(dd x) {
  float y = rcp_approx(x.hi);
  y = __fmaf_rn(y, __fmaf_rn(-x.hi, y, 1.f), y);
  const float e = __fmaf_rn(-x.lo, y, __fmaf_rn(-x.hi, y, 1.f));
  return dd_fast_two_sum(y, __fmul_rn(y, __fmaf_rn(e, e, e)));
}
__device__ __forceinline__ dd unit_rsqrt(dd x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x.hi));
  y = __fmaf_rn(__fmul_rn(0.5f, y), __fmaf_rn(-__fmul_rn(x.hi, y), y, 1.f), y);
  const dd y2 = dd_two_prod(y, y);
  const dd t = x * y2;                               // 1 - e
  const float e = __fsub_rn(__fsub_rn(1.f, t.hi), t.lo);
  return dd_fast_two_sum(y, __fmul_rn(__fmul_rn(y, e), __fmaf_rn(0.375f, e, 0.5f)));
}

// psi of Eqs. EOS and InteractionPotential; rho <= 0 is non-physical as well as psi^2 < 0 or NaN.
// FP32 pairs: without a branch - one would cut the rows of a walk apart for the instruction
// scheduler.
__device__ __forceinline__ f2 unit_psi(f2 rho, f2 k1, f2, const UnitT<f2>& k, int& flag) {
  const f2 one = cst<f2>(1.0);
  const f2 eta = k.p.b4 * rho;
  const f2 om = one - eta;
  const f2 num = fmadd(eta, fmadd(eta, om, one), one);  // 1 + eta + eta^2 - eta^3
  const f2 q = num * unit_rcp(om * om * om);
  const f2 p2 = rho * fmadd(k1, q, fmadd(k.p.k2, rho, k.p.k3));
  const float s = lo(p2), t = hi(p2);
  if (!(s >= 0.f && t >= 0.f && lo(rho) > 0.f && hi(rho) > 0.f)) flag |= STATUS_NONPHYS;
  return make_f2(sqrt_approx(fmaxf(s, 0.f)), sqrt_approx(fmaxf(t, 0.f)));
}
__device__ __forceinline__ double unit_psi(double rho, double k1, double, const UnitT<double>& k, int& flag) {
  if (nonpositive(rho)) flag |= STATUS_NONPHYS;
  return psi_k1(rho, k1, k.p, flag);
}
__device__ __forceinline__ dd unit_psi(dd rho, dd k1, dd RT, const UnitT<dd>& k, int& flag) {
  const dd one = cst<dd>(1.0);
  const dd eta = k.p.b4 * rho;
  const dd om = one - eta;
  const dd num = fmadd(eta, fmadd(eta, om, one), one);
  const dd D = om * om * om;
  const dd N = rho * fmadd(fmadd(k.p.k2, rho, k.p.k3), D, k1 * num);
  if (N.hi > 0.f && D.hi > 0.f && rho.hi > 0.f) return N * unit_rsqrt(N * D);
  if (nonpositive(rho)) flag |= STATUS_NONPHYS;
  return psi_k1(rho, k1, k.p, flag);
}

// the post-collision values o of a node with moments (dr, jx, jy) before the collision, the
// potential psi and the stencil sums (Sx, Sy) (zero on wall rows); dmean = <rho> - rho_ref
template <typename V>
struct Velocity {
  V rho, ux, uy;
};
// FORM 1, 2: the gravity of Eq. Gravity_1, Eq. Gravity_2; 0: either, with rho_ref or
// -(<rho> - rho_ref) in the place of dmean
template <int FORM, typename V>
__device__ __forceinline__ Velocity<V> unit_velocity(V dr, V jx, V jy, V psi, V Sx, V Sy, V dmean, const UnitT<V>& k,
                                                     V& Fx, V& Fy) {
  const V rho = k.p.rho_ref + dr;
  const V base = FORM == 2 ? dr - dmean : (FORM == 1 ? rho : dr + dmean);
  const V t = k.p.negG * psi;
  Fx = fmadd(t, Sx, base * k.p.gx);
  Fy = fmadd(t, Sy, base * k.p.gy);
  const V inv = unit_rcp(rho);
  return {rho, fma2(0.5, Fx, jx) * inv, fma2(0.5, Fy, jy) * inv};  // Eq. Momentum
}
// double-float: products only by 1/9 and 1/3, the other factors are powers of two
__device__ __forceinline__ void unit_back(dd dr, dd jx, dd jy, dd A36, dd pxx, dd pq, dd (&o)[9]) {
  const dd d9 = cst<dd>(1.0 / 9.0) * dr;
  o[0] = scale2(4.0, d9) - scale2(8.0, A36);
  const dd ba = d9 + A36, bd = scale2(0.25, d9) + A36;
  const dd q = scale2(0.25, pxx), r = scale2(0.125, pq);
  const dd tp = ba + q, tm = ba - q, up = bd + r, um = bd - r;
  const dd x3 = cst<dd>(1.0 / 3.0) * jx, y3 = cst<dd>(1.0 / 3.0) * jy;
  o[1] = tp + x3;
  o[3] = tp - x3;
  o[2] = tm + y3;
  o[4] = tm - y3;
  const dd s = scale2(0.25, x3 + y3), t = scale2(0.25, y3 - x3);
  o[5] = up + s;
  o[7] = up - s;
  o[6] = um + t;
  o[8] = um - t;
}

template <int FORM, typename V>
__device__ __forceinline__ Velocity<V> unit_collide(V dr, V jx, V jy, V psi, V Sx, V Sy, V dmean, const UnitT<V>& k,
                                                    V (&o)[9]) {
  V Fx, Fy;
  const Velocity<V> u = unit_velocity<FORM>(dr, jx, jy, psi, Sx, Sy, dmean, k, Fx, Fy);
  const V jsx = jx + Fx, jsy = jy + Fy;                       // j*
  const V hx = fma2(0.5, Fx, jsx), hy = fma2(0.5, Fy, jsy);   // rho u + F
  const V a = u.ux * hx, b = u.uy * hy;
  const V pq = fmadd(u.ux, hy, u.uy * hx);                    // 2 p_xy*
  const V S2 = fmadd(Sx, Sx, Sy * Sy);
  const V A36 = fmadd(cst<V>(1.0 / 12.0), a + b, k.p.kS * S2);  // A/36
  unit_back(dr, jsx, jsy, A36, a - b, pq, o);
  return u;
}

// Zou-He wall node (Sec. III): K counts the known populations as zou_he() does; the node's
// density deviation, and j = -F_g/2 so that the velocity vanishes
template <typename V>
__device__ __forceinline__ void unit_zou_he(V K, bool bottom, V dmean, const UnitT<V>& k, V& dr, V& jx, V& jy) {
  const V sg = (bottom ? cst<V>(0.5) : cst<V>(-0.5)) * k.p.gy;
  const V num = (k.p.form == 2) ? fmadd(sg, dmean, K) : K - sg * k.p.rho_ref;
  // num/(1 + s) = num - num s/(1 + s): s is small, so its rounding does not move the density the
  // same way at every step, as a rounded factor 1/(1 + s) would
  dr = fmadd(cst<V>(-1.0) * fast_div(sg, cst<V>(1.0) + sg), num, num);
  const V base = (k.p.form == 2) ? (dr - dmean) : (k.p.rho_ref + dr);
  const V mh = cst<V>(-0.5);
  jx = mh * (base * k.p.gx);
  jy = mh * (base * k.p.gy);
}

}  // namespace lbm
