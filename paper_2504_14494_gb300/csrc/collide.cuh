// Collisions shared by the single-step and the multi-step kernels: the channel
// node, and the BGK collision of common.cuh for two nodes at a time.
#pragma once
#include "common.cuh"

namespace lbmgnn {

// Correctly rounded 1/x for |x| in [2^-100, 2^100] by Markstein's method ("Computation of
// elementary functions on the IBM RISC System/6000 processor", 1990): the residual of the
// hardware's approximate reciprocal, exact in one FMA, corrects it in a second one.  Equal to
// 1.0f / x for every float of that range (all 2^24 x 201 compared on the GPU).
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

// bgk_collide() of 2 NP nodes in packed FP32 pairs (one instruction for two
// nodes), nomega = -1/tau: the same roundings in the same order as the
// compiler makes of bgk_collide (products contracted into the following
// addition; 1.5 u.u stays a product and is contracted into each direction's
// sum), so the results are equal bit for bit, non-finite ones included: a
// non-finite velocity makes every population NaN there through 0 * u, which
// `poison` carries into the common sum here.
template <int NP>
__device__ __forceinline__ void bgk_collide_pairs(float2 (&f)[Q][NP], float2 nomega) {
  auto c2 = [](float v) { return make_float2(v, v); };
  auto sub = [&](float2 a, float2 b) { return __ffma2_rn(b, c2(-1.0f), a); };
  float2 rho[NP], inv[NP];
#pragma unroll
  for (int c = 0; c < NP; ++c) {
    rho[c] = __fadd2_rn(__fadd2_rn(__fadd2_rn(f[0][c], __fadd2_rn(f[1][c], f[3][c])),
                                   __fadd2_rn(f[2][c], f[4][c])),
                        __fadd2_rn(__fadd2_rn(f[5][c], f[7][c]), __fadd2_rn(f[6][c], f[8][c])));
    inv[c] = rcp2_mid(rho[c]);
  }
  bool mid = true;  // (false for a NaN)
#pragma unroll
  for (int c = 0; c < NP; ++c)
    mid = mid && rho[c].x >= 0x1p-90f && rho[c].x <= 0x1p90f && rho[c].y >= 0x1p-90f &&
          rho[c].y <= 0x1p90f;
  if (!mid) {
#pragma unroll
    for (int c = 0; c < NP; ++c) inv[c] = make_float2(1.0f / rho[c].x, 1.0f / rho[c].y);
  }
#pragma unroll
  for (int c = 0; c < NP; ++c) {
    const float2 d57 = sub(f[5][c], f[7][c]), d86 = sub(f[8][c], f[6][c]);
    const float2 jx = __fadd2_rn(__fadd2_rn(sub(f[1][c], f[3][c]), d57), d86);
    const float2 jy = sub(__fadd2_rn(sub(f[2][c], f[4][c]), d57), d86);
    const float2 ux = __fmul2_rn(jx, inv[c]), uy = __fmul2_rn(jy, inv[c]);
    const float2 poison = __ffma2_rn(c2(0.0f), ux, __fmul2_rn(c2(0.0f), uy));
    const float2 usq = __fadd2_rn(__ffma2_rn(ux, ux, __fmul2_rn(uy, uy)), poison);
    auto relax = [&](int q, float2 t, float2 nwr) {
      t = __ffma2_rn(c2(-1.5f), usq, t);
      f[q][c] = __ffma2_rn(nomega, __ffma2_rn(nwr, t, f[q][c]), f[q][c]);
    };
    auto both = [&](int q, int o, float2 eu, float2 nwr) {  // direction q and its opposite o
      const float2 a = __fmul2_rn(c2(4.5f), eu);
      relax(q, __ffma2_rn(a, eu, __ffma2_rn(c2(3.0f), eu, c2(1.0f))), nwr);
      relax(o, __ffma2_rn(a, eu, __ffma2_rn(c2(-3.0f), eu, c2(1.0f))), nwr);
    };
    const float2 w1 = __fmul2_rn(c2(-wq(1)), rho[c]), w5 = __fmul2_rn(c2(-wq(5)), rho[c]);
    relax(0, c2(1.0f), __fmul2_rn(c2(-wq(0)), rho[c]));
    both(1, 3, ux, w1);
    both(2, 4, uy, w1);
    both(5, 7, __fadd2_rn(ux, uy), w5);
    both(6, 8, sub(uy, ux), w5);
  }
}

// bgk_collide() of one node, the same way as bgk_collide_pairs.
__device__ __forceinline__ void bgk_collide_one(float (&f)[Q], float omega) {
  const float rho = __fadd_rn(
      __fadd_rn(__fadd_rn(f[0], __fadd_rn(f[1], f[3])), __fadd_rn(f[2], f[4])),
      __fadd_rn(__fadd_rn(f[5], f[7]), __fadd_rn(f[6], f[8])));
  const float inv = rcp1(rho);
  const float d57 = __fsub_rn(f[5], f[7]), d86 = __fsub_rn(f[8], f[6]);
  const float ux = __fmul_rn(__fadd_rn(__fadd_rn(__fsub_rn(f[1], f[3]), d57), d86), inv);
  const float uy = __fmul_rn(__fsub_rn(__fadd_rn(__fsub_rn(f[2], f[4]), d57), d86), inv);
  const float poison = __fmaf_rn(0.0f, ux, __fmul_rn(0.0f, uy));
  const float usq = __fadd_rn(__fmaf_rn(ux, ux, __fmul_rn(uy, uy)), poison);
  auto relax = [&](int q, float t, float nwr) {
    t = __fmaf_rn(-1.5f, usq, t);
    f[q] = __fmaf_rn(-omega, __fmaf_rn(nwr, t, f[q]), f[q]);
  };
  auto both = [&](int q, int o, float eu, float nwr) {
    const float a = __fmul_rn(4.5f, eu);
    relax(q, __fmaf_rn(a, eu, __fmaf_rn(3.0f, eu, 1.0f)), nwr);
    relax(o, __fmaf_rn(a, eu, __fmaf_rn(-3.0f, eu, 1.0f)), nwr);
  };
  const float w1 = __fmul_rn(-wq(1), rho), w5 = __fmul_rn(-wq(5), rho);
  relax(0, 1.0f, __fmul_rn(-wq(0), rho));
  both(1, 3, ux, w1);
  both(2, 4, uy, w1);
  both(5, 7, __fadd_rn(ux, uy), w5);
  both(6, 8, __fsub_rn(uy, ux), w5);
}

// f_i - (f_i - f_i^eq(rho, u))/t + (1 - 1/(2t)) w_i [3 (e_i - u) + 9 (e_i.u) e_i].(gx, 0)
// with u the force-corrected velocity; t is tau (BGK) or tau tau_adj (Eq. 3).
__device__ __forceinline__ void channel_relax(float (&f)[Q], float t, float gx) {
  const float rho = ((f[0] + (f[1] + f[3])) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8]));
  const float jx = (f[1] - f[3]) + (f[5] - f[7]) + (f[8] - f[6]);
  const float jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
  const float inv = rcp1(rho);
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
