// Collisions shared by the single-step, the batched and the multi-step kernels.
// In the BGK collision every rounding is spelled out (the _rn intrinsics are not
// contracted by the compiler), so that each kernel, whatever else it does, gives
// a node the same bits, and one formula serves a node and a packed pair of nodes.
#pragma once
#include "common.cuh"

namespace lbmgnn {

// Arithmetic on one value, and on two in packed FP32 instructions.
struct One {
  using T = float;
  static __device__ __forceinline__ T c(float v) { return v; }
  static __device__ __forceinline__ T add(T a, T b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ T sub(T a, T b) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ T mul(T a, T b) { return __fmul_rn(a, b); }
  static __device__ __forceinline__ T fma(T a, T b, T d) { return __fmaf_rn(a, b, d); }
};
struct Two {
  using T = float2;
  static __device__ __forceinline__ T c(float v) { return make_float2(v, v); }
  static __device__ __forceinline__ T add(T a, T b) { return __fadd2_rn(a, b); }
  static __device__ __forceinline__ T sub(T a, T b) { return __ffma2_rn(b, c(-1.0f), a); }
  static __device__ __forceinline__ T mul(T a, T b) { return __fmul2_rn(a, b); }
  static __device__ __forceinline__ T fma(T a, T b, T d) { return __ffma2_rn(a, b, d); }
};

// Correctly rounded 1/x for |x| in [2^-100, 2^100] by Markstein's method ("Computation of
// elementary functions on the IBM RISC System/6000 processor", 1990): the residual of the
// hardware's approximate reciprocal, exact in one FMA, corrects it in a second one.  Equal to
// 1.0f / x for every float of that range (lbm_selftest_reciprocal compares them all).
__device__ __forceinline__ float2 rcp2_mid(float2 x) {
  float2 r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(x.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(x.y));
  const float2 e = __ffma2_rn(make_float2(-x.x, -x.y), r, make_float2(1.0f, 1.0f));
  return __ffma2_rn(r, e, r);
}

// The same for one value, any x.
__device__ __forceinline__ float rcp1(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  r = __fmaf_rn(r, __fmaf_rn(-x, r, 1.0f), r);
  if (!(x >= 0x1p-90f && x <= 0x1p90f)) r = 1.0f / x;
  return r;
}

// Density and momentum sums of pulled populations.
template <class A>
__device__ __forceinline__ typename A::T rho9(const typename A::T (&f)[Q]) {
  return A::add(A::add(A::add(f[0], A::add(f[1], f[3])), A::add(f[2], f[4])),
                A::add(A::add(f[5], f[7]), A::add(f[6], f[8])));
}
template <class A>
__device__ __forceinline__ void mom9(const typename A::T (&f)[Q], typename A::T& jx,
                                     typename A::T& jy) {
  const auto d57 = A::sub(f[5], f[7]), d86 = A::sub(f[8], f[6]);
  jx = A::add(A::add(A::sub(f[1], f[3]), d57), d86);
  jy = A::sub(A::add(A::sub(f[2], f[4]), d57), d86);
}
// u.u.  A non-finite velocity makes every population NaN (as 0 * u_x in e.u
// does where e_x = 0): the two products by 0 carry it into the common sum.
template <class A>
__device__ __forceinline__ typename A::T usq9(typename A::T ux, typename A::T uy) {
  const auto zero = A::fma(A::c(0.0f), ux, A::mul(A::c(0.0f), uy));
  return A::add(A::fma(ux, ux, A::mul(uy, uy)), zero);
}
// 1 + 3 e.u + 9/2 (e.u)^2 - 3/2 u.u of direction sign * e, eu = e.u, e45 = 4.5 eu.
template <class A>
__device__ __forceinline__ typename A::T feq_poly(float sign, typename A::T eu, typename A::T e45,
                                                  typename A::T usq) {
  const auto t = A::fma(e45, eu, A::fma(A::c(3.0f * sign), eu, A::c(1.0f)));
  return A::fma(A::c(-1.5f), usq, t);
}

// BGK collision (Eq. 1 with Eq. 2) in place, given rho, 1/rho and -1/tau:
// f_i - (1/tau) (f_i - rho w_i (1 + 3 e.u + 9/2 (e.u)^2 - 3/2 u.u)).
template <class A>
__device__ __forceinline__ void bgk_relax(typename A::T (&f)[Q], typename A::T rho,
                                          typename A::T inv, typename A::T nomega) {
  using T = typename A::T;
  T jx, jy;
  mom9<A>(f, jx, jy);
  const T ux = A::mul(jx, inv), uy = A::mul(jy, inv), usq = usq9<A>(ux, uy);
  auto relax = [&](int q, T t, T nwr) { f[q] = A::fma(nomega, A::fma(nwr, t, f[q]), f[q]); };
  auto both = [&](int q, int o, T eu, T nwr) {  // direction q and its opposite o
    const T e45 = A::mul(A::c(4.5f), eu);
    relax(q, feq_poly<A>(1.0f, eu, e45, usq), nwr);
    relax(o, feq_poly<A>(-1.0f, eu, e45, usq), nwr);
  };
  const T w1 = A::mul(A::c(-wq(1)), rho), w5 = A::mul(A::c(-wq(5)), rho);
  relax(0, A::fma(A::c(-1.5f), usq, A::c(1.0f)), A::mul(A::c(-wq(0)), rho));
  both(1, 3, ux, w1);
  both(2, 4, uy, w1);
  both(5, 7, A::add(ux, uy), w5);
  both(6, 8, A::sub(uy, ux), w5);
}

// One node; omega = 1/tau.
__device__ __forceinline__ void bgk_collide(float (&f)[Q], float omega) {
  const float rho = rho9<One>(f);
  bgk_relax<One>(f, rho, 1.0f / rho, -omega);
}
// One node with the reciprocal that does not branch apart (multi_step.cu).
__device__ __forceinline__ void bgk_collide_fast(float (&f)[Q], float omega) {
  const float rho = rho9<One>(f);
  bgk_relax<One>(f, rho, rcp1(rho), -omega);
}
// Two nodes; nomega = -1/tau.
__device__ __forceinline__ void bgk_collide_pair(float2 (&f)[Q], float2 nomega) {
  const float2 rho = rho9<Two>(f);
  float2 inv = rcp2_mid(rho);
  if (!(rho.x >= 0x1p-90f && rho.x <= 0x1p90f && rho.y >= 0x1p-90f && rho.y <= 0x1p90f))
    inv = make_float2(1.0f / rho.x, 1.0f / rho.y);
  bgk_relax<Two>(f, rho, inv, nomega);
}

// f_i - (f_i - f_i^eq(rho, u))/t + (1 - 1/(2t)) w_i [3 (e_i - u) + 9 (e_i.u) e_i].(gx, 0)
// with u the force-corrected velocity; t is tau (BGK) or tau tau_adj (Eq. 3).
// (Its contractions are the compiler's: spelled out, in four forms with the same
// bits, 2,000 steps of a 4 x 32 channel took 457 to 561 us instead of 447.)
// FAST: the reciprocal without the division's length in the chain, for the steps
// on chip; a single step, bound by memory, takes the division (2048^2 71.9 us
// against 72.6, in a row of calls 73.9 against 75.6).
template <bool FAST>
__device__ __forceinline__ void channel_relax(float (&f)[Q], float t, float gx) {
  const float rho = ((f[0] + (f[1] + f[3])) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8]));
  const float jx = (f[1] - f[3]) + (f[5] - f[7]) + (f[8] - f[6]);
  const float jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
  const float inv = FAST ? rcp1(rho) : 1.0f / rho;
  const Moments m{rho, (jx + 0.5f * gx) * inv, jy * inv};
  const float usq15 = 1.5f * (m.ux * m.ux + m.uy * m.uy);
  const float omega = 1.0f / t, pre = 1.0f - 0.5f * omega;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const float eu = float(ex(q)) * m.ux + float(ey(q)) * m.uy;
    const float src = pre * wq(q) * (3.0f * (float(ex(q)) - m.ux) + 9.0f * eu * float(ex(q))) * gx;
    f[q] = f[q] - omega * (f[q] - feq_i(q, m, usq15)) + src;
  }
}

}  // namespace lbmgnn
