// GNN-enhanced collision, reverse direction and training (paper Sec. 2.4,
// Eq. 3, Eq. 4): the Eq. 3 + MSE loss kernel, the head backward, the two
// kernels of each message-passing round's backward, the encoder backward,
// the deterministic gradient reduction and the AdamW update.
//
// Per-round recompute: the forward saves h, the aggregated messages a and
// the per-node edge terms A = W_a h, B = W_b h (FP16); the backward recomputes
// the node pre-activation W_n [h; a] + b_n with the same MMA and every edge
// pre-activation z_ik = A_i + B_j + c_k elementwise, so the 8 per-node edge
// activations are never stored.
//
// The edge terms need gradients scattered to neighbours (dB_j collects from
// every i with j = i + e_k).  They are gathered instead ("pull" form): node j
// reads da_i and A_i of its 8 neighbours i = j - e_k, so no atomics are used
// and the result is deterministic.  This needs da of every node first, hence
// two kernels per round.
//
// Weight gradients are contractions over nodes.  Each CTA accumulates them
// on the tensor cores over all tiles it owns (FP32 accumulators in tensor
// memory) and writes one partial row; a final kernel sums the rows in a fixed
// order.  Their operands are the node-major tiles of the other products, read
// across their rows (umma.cuh, MN-major): no transposed copies.  Bias gradients
// (column sums) ride along as an extra MMA column of ones.
#include "gnn.cuh"
#include "gnn_launch.h"
#include "launch.h"

namespace lbmgnn {

// ---- transposed operand writes ---------------------------------------------------
// Writes NV values v[c] to rows row0 + c, column `node` (0..127) of a K = 128
// operand made of two SW128 blocks of R rows each (nodes 0..63, 64..127).
template <int NV>
__device__ __forceinline__ void st_col(uint8_t* op, int R, int row0, int node, const float* v) {
  uint8_t* blk = op + (node >> 6) * (R * 128);
  const int k = node & 63;
#pragma unroll
  for (int c = 0; c < NV; ++c)
    *reinterpret_cast<__nv_bfloat16*>(blk + sw128_off(row0 + c, k)) = __float2bfloat16_rn(v[c]);
}

// Features f0..f0+NF-1 of node n, BF16 words as they are, into row `row` of an
// SW128 block.
template <int NF, bool PREV = false>
__device__ __forceinline__ void copy_row(uint8_t* blk, int row, int f0, const __nv_bfloat16* base,
                                         int64_t N, int64_t n) {
#pragma unroll
  for (int c = 0; c < NF / 8; ++c) {
    const int chunk = (f0 >> 3) + c;
    *reinterpret_cast<uint4*>(blk + row * 128 + ((chunk ^ (row & 7)) << 4)) =
        ld_in<PREV>(chunk8(base, N, n, f0 + 8 * c));
  }
}

// Part [off, off + n) of a partial gradient row set to 0 (a CTA whose
// tensor-core wait gave up).
__device__ __forceinline__ void zero_grad(float* g, int off, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) g[off + i] = 0.0f;
}

#ifndef LBM_BWD_PF
#define LBM_BWD_PF 1  // L2 prefetch of the next tile's per-node inputs
#endif

// L2 prefetch (a hint: no registers, no completion to wait for) of nodes
// [m0, m0 + 128) of plane `plane` of a per-node tensor: chunked planes of 16
// bytes per node (esz 16, plane stride N nodes) or FP32 planes (esz 4, plane
// stride `ps` nodes).  The range is shrunk to 16-byte boundaries inside the
// tensor's own bytes.
__device__ __forceinline__ void l2_prefetch_nodes(const void* base, int plane, int64_t ps,
                                                  int esz, int64_t m0, int64_t N) {
  if (m0 >= N) return;
  const int64_t cnt = N - m0 < 128 ? N - m0 : 128;
  const uintptr_t a = reinterpret_cast<uintptr_t>(base) + (uintptr_t)((plane * ps + m0) * esz);
  const uintptr_t lo = a & ~uintptr_t(15), hi = (a + (uintptr_t)(cnt * esz)) & ~uintptr_t(15);
  if (hi > lo)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"((uint32_t)(hi - lo))
                 : "memory");
}

__device__ __forceinline__ void zero_smem(uint8_t* p, uint32_t bytes) {
  uint4* q = reinterpret_cast<uint4*>(p);
  for (uint32_t i = threadIdx.x; i < bytes / 16; i += blockDim.x) q[i] = make_uint4(0, 0, 0, 0);
}

// Sets row `row` of a two-block K = 128 operand (R rows per block) to 1.
__device__ __forceinline__ void ones_row(uint8_t* op, int R, int row) {
  for (int n = threadIdx.x; n < 128; n += blockDim.x) {
    uint8_t* blk = op + (n >> 6) * (R * 128);
    *reinterpret_cast<__nv_bfloat16*>(blk + sw128_off(row, n & 63)) = __float2bfloat16_rn(1.0f);
  }
}

// Sum over the 32 lanes of v[0..31] (lane-private values): afterwards lane l
// holds the sum of v[l] over the warp (31 shuffles; halves the vector per step).
__device__ __forceinline__ float warp_transpose_sum(float (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int w = 16; w >= 1; w >>= 1) {
    const bool upper = lane & w;  // keep the upper half of the current range
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float send = upper ? v[i] : v[i + w];
      const float keep = upper ? v[i + w] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
    }
  }
  return v[0];
}

__device__ __forceinline__ void ld_f32x32(const float* p, float* v) {
  const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 t = __ldg(q + i);
    v[4 * i] = t.x;
    v[4 * i + 1] = t.y;
    v[4 * i + 2] = t.z;
    v[4 * i + 3] = t.w;
  }
}
__device__ __forceinline__ void st_f32x32(float* p, const float* v) {
  float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
  for (int i = 0; i < 8; ++i) q[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
}

// ---------------------------------------------------------------------------
// Eq. 3 followed by Eq. 4: per node f_pred = f - (f - f_eq)/(tau tau_adj) +
// s_df y_1..9, squared error against the target, and dL/dy.  The loss is the
// mean over nodes x 9 of the whole stack.  One thread per node.
// FORCED (the channel): a force (gx, 0) per unit volume (gxs[b] per lattice
// when set) enters by Guo's scheme, u = (sum f e + F/2)/rho and the source
// (1 - 1/(2t)) S with S_i = w_i [3 (e_ix - u_x) + 9 (e_i.u) e_ix] gx at the
// network's time t; d f_pred / d t = ((f - f_eq) + S/2) / t^2.
template <bool FORCED>
__global__ void __launch_bounds__(256) gnn_collide_loss_kernel(
    const float* f_pre, const float* y, const float* tgt, Shape s, float tau, const float* taus,
    float gx0, const float* gxs, const uint8_t* packed, double* __restrict__ lossp,
    float* __restrict__ dy, float* __restrict__ f_pred, const float* lw, unsigned* stw) {
  dep_sync();
  packed = after_wait(packed);
  if (!blob_ok(packed, stw)) {  // no loss from an invalid image: NaN
    if (threadIdx.x == 0) lossp[blockIdx.x] = __longlong_as_double(0x7ff8000000000000LL);
    return;
  }
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const int64_t n = after_wait((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  const bool on = n < N;
  const int64_t nn = on ? n : N - 1;
  const float sdf = reinterpret_cast<const float*>(packed + K::NORM)[24];
  const int variant = variant_of(reinterpret_cast<const float*>(packed + K::NORM));
  float fv[Q], yv[NOUT];
#pragma unroll
  for (int q = 0; q < Q; ++q) fv[q] = ld_prev(f_pre + q * s.ps + nn);
#pragma unroll
  for (int o = 0; o < NOUT; ++o) yv[o] = ld_prev(y + o * N + nn);
  const int64_t b = nn / ((int64_t)s.nx * s.ny);
  const float t = taus ? ld_prev(taus + b) : tau;
  const float wb = lw ? ld_prev(lw + b) : 1.0f;  // per-instance loss weight (1: Eq. 4)
  Moments m = moments9(fv);
  float gx = 0.0f;
  if constexpr (FORCED) {
    gx = gxs ? ld_prev(gxs + b) : gx0;
    m.ux += 0.5f * gx / m.rho;
  }
  const float usq15 = 1.5f * (m.ux * m.ux + m.uy * m.uy);
  const bool fixed_tau = variant & VAR_FIXED_TAU;
  const float sg = sigmoid_acc(yv[0]);
  const float teff = t * tau_adj_of(yv[0], variant);
  const float inv = 1.0f / teff;
  const float scale = 2.0f * wb / (9.0f * (float)N);
  float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;  // sum of r^2, unevaluated
  float dta = 0.0f, dyv[NOUT], d[Q], g[Q], rr[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) d[q] = sdf * yv[1 + q];
  if (variant & VAR_CONSERVATIVE) conserve9(d);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const float fe = feq_i(q, m, usq15);
    float fp = fv[q] - (fv[q] - fe) * inv + d[q];
    float dt = fv[q] - fe;  // t^2 d f_pred / d t
    if constexpr (FORCED) {
      const float eu = float(ex(q)) * m.ux + float(ey(q)) * m.uy;
      const float src = wq(q) * (3.0f * (float(ex(q)) - m.ux) + 9.0f * eu * float(ex(q))) * gx;
      fp += (1.0f - 0.5f * inv) * src;
      dt += 0.5f * src;
    }
    const float r = fp - ld_prev(tgt + q * s.ps + nn);
    rr[q] = r;
    // r^2 = r2 + fma(r, r, -r2) exactly; the first two sums are error-free
    const float r2 = __fmul_rn(r, r);
    float e, f;
    two_sum(s0, r2, s0, e);
    two_sum(s1, e, s1, e);
    two_sum(s1, __fmaf_rn(r, r, -r2), s1, f);
    s2 = __fadd_rn(s2, __fadd_rn(e, f));
    g[q] = scale * r;  // dL/df*
    dta += g[q] * dt;
    if (on && f_pred) f_pred[q * s.ps + n] = fp;
  }
  // The squared error goes on in FP64.  The node's sum S of r^2 was carried in
  // three FP32 words: s0 and s1 take error-free sums, |s1| <= 18 2^-24 S,
  // |s2| <= 18 2^-24 |s1|, and the 18 additions into s2 round, which is below
  // 2^-59 S in all; with the addition and the weight's product here the node's
  // value is within 2.1 2^-53.  Nine FP64 products and sums, within 10 2^-53,
  // bound the call (4.2 M nodes, with the finish: 311 us against 169); they are
  // used where r^2 leaves the range in which its rounding error is an FP32
  // number.
  double lp = (double)s0 + ((double)s1 + (double)s2);
  if (lw) lp *= (double)wb;
  if (!(s0 >= 1e-25f && s0 < 1e30f)) {
    lp = 0.0;
#pragma unroll
    for (int q = 0; q < Q; ++q) lp += (double)wb * (double)rr[q] * (double)rr[q];
  }
  // Delta f = s_df P y_1..9 with P the (symmetric) projection, or P = I
  if (variant & VAR_CONSERVATIVE) conserve9(g);
#pragma unroll
  for (int q = 0; q < Q; ++q) dyv[1 + q] = sdf * g[q];
  dyv[0] = fixed_tau ? 0.0f : dta * t * inv * inv * sg * (1.0f - sg);
  if (on && dy) {
#pragma unroll
    for (int o = 0; o < NOUT; ++o) dy[o * N + n] = dyv[o];
  }
  if (!on) lp = 0.0;
  __shared__ double red[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lp += __shfl_xor_sync(0xffffffffu, lp, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = lp;
  __syncthreads();
  if (threadIdx.x == 0) {
    double acc = 0.0;
    for (int i = 0; i < 8; ++i) acc += red[i];
    lossp[blockIdx.x] = acc;
  }
}

// Reverse mode of Eq. 3 for the K-step rollout loss, one thread per node:
// g = g_in + scale (f_post - target) is dL/df* of this step (g_in: the
// later steps' share, pulled back through streaming; NULL for the last
// step); writes dL/dy as the loss kernel does and the part of dL/df_pre that
// passes through the explicit f and f^eq(rho(f), u(f)):
//   dfd_j = g_j (1 - 1/t) + (1/t) [sum_i g_i f^eq_i / rho
//           + V . (e_j - u)],  V = sum_i g_i w_i (3 e_i + 9 (e_i.u) e_i - 3 u).
__global__ void __launch_bounds__(256) gnn_collide_adjoint_kernel(
    const float* __restrict__ f_pre, const float* __restrict__ y,
    const float* __restrict__ f_post, const float* __restrict__ tgt,
    const float* g_in, Shape s, float tau, const float* __restrict__ taus,
    const uint8_t* __restrict__ packed, float scale, float* __restrict__ dy,
    float* __restrict__ dfd, unsigned* stw) {
  dep_sync();
  if (!blob_ok(packed, stw)) return;
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const int64_t n = after_wait((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  if (n >= N) return;
  const float* nrm = reinterpret_cast<const float*>(packed + K::NORM);
  const float sdf = nrm[24];
  const int variant = variant_of(nrm);
  float fv[Q], g[Q], gp[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    fv[q] = __ldg(f_pre + q * s.ps + n);
    const float r = __ldg(f_post + q * s.ps + n) - __ldg(tgt + q * s.ps + n);
    g[q] = (g_in ? ld_prev(g_in + q * s.ps + n) : 0.0f) + scale * r;
    gp[q] = g[q];
  }
  const float y0 = __ldg(y + n);
  const int64_t b = n / ((int64_t)s.nx * s.ny);
  const float t0 = taus ? __ldg(taus + b) : tau;
  const float sg = sigmoid_acc(y0);
  const float t = t0 * tau_adj_of(y0, variant);
  const float inv = 1.0f / t;
  const Moments m = moments9(fv);
  const float usq15 = 1.5f * (m.ux * m.ux + m.uy * m.uy);
  float dta = 0.0f, a = 0.0f, vx = 0.0f, vy = 0.0f;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const float fe = feq_i(q, m, usq15);
    dta += g[q] * (fv[q] - fe);
    a += g[q] * fe;
    const float eu = float(ex(q)) * m.ux + float(ey(q)) * m.uy;
    const float gw = g[q] * wq(q);
    vx += gw * (3.0f * float(ex(q)) + 9.0f * eu * float(ex(q)) - 3.0f * m.ux);
    vy += gw * (3.0f * float(ey(q)) + 9.0f * eu * float(ey(q)) - 3.0f * m.uy);
  }
  a /= m.rho;
  if (variant & VAR_CONSERVATIVE) conserve9(gp);
#pragma unroll
  for (int q = 0; q < Q; ++q) dy[(int64_t)(1 + q) * N + n] = sdf * gp[q];
  dy[n] = (variant & VAR_FIXED_TAU) ? 0.0f : dta * t0 * inv * inv * sg * (1.0f - sg);
#pragma unroll
  for (int q = 0; q < Q; ++q)
    dfd[q * s.ps + n] = g[q] * (1.0f - inv) +
                        inv * (a + vx * (float(ex(q)) - m.ux) + vy * (float(ey(q)) - m.uy));
}

// Adjoint of periodic pull streaming applied to a + b: out_q(x) =
// (a + b)_q(x + e_q) within each lattice (the transpose of
// f_q(x) = f*_q(x - e_q)).
__global__ void __launch_bounds__(256) stream_adjoint_sum_kernel(
    const float* __restrict__ a, const float* __restrict__ b, float* __restrict__ out, Shape s,
    unsigned* stw) {
  dep_sync();
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const NodeXY p = node_xy(n, s);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int64_t j = checked(node_at(p, ex(q), ey(q), s), 0, N, stw);
    out[q * s.ps + n] = __ldg(a + q * s.ps + j) + __ldg(b + q * s.ps + j);
  }
}

// Sum of the per-block squared errors, divided by 9 N (deterministic order).
// One block: 1,024 threads with 8 loads in flight each (34 us for 16,384
// values with 256 threads and one load at a time).
__global__ void __launch_bounds__(1024) loss_finish_kernel(const double* lossp, int nblk,
                                                           double count,
                                                           double* __restrict__ loss) {
  dep_sync();
  __shared__ double red[32];
  double acc = 0.0;
#pragma unroll 8
  for (int i = after_wait((int)threadIdx.x); i < nblk; i += 1024) acc += ld_prev(lossp + i);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc = red[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (threadIdx.x == 0) *loss = acc / count;
  }
}

// ---------------------------------------------------------------------------
// Head backward: dh2 = dy W_h (CUDA cores), dW_h and db_h accumulated on the
// tensor cores: D[o][i] += sum_n dy[n][o] [h2 | 1][n][i].
namespace hb {
// XT: dy transposed (128 rows, 10 used), H2: h2 node-major, ONE: 16 rows, row 0 ones
constexpr uint32_t XT = 0, ONE = 32768, H2 = 36864, WHF = 53248, DYS = 55808, SH = 60928,
                   BYTES = 61056;
}

#ifndef LBM_HB_CTAS
#define LBM_HB_CTAS 2  // resident CTAs per SM
#endif
__global__ void __launch_bounds__(256, LBM_HB_CTAS) gnn_head_bwd_kernel(
    const float* dy, const __nv_bfloat16* h2, float* __restrict__ dh, float* __restrict__ G,
    Shape s, const uint8_t* packed, unsigned* stw) {
  dep_wait();  // before the weights: as a call's first kernel it may follow their pack
  packed = after_wait(packed);
  if (!blob_ok(packed, stw)) return;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = smem_align1024(smem_raw);
  TcShared* sh = reinterpret_cast<TcShared*>(sm + hb::SH);
  zero_smem(sm, hb::H2);
  copy_g2s<true>(sm + hb::WHF, packed + K::WHF, 2560);
  __syncthreads();
  ones_row(sm + hb::ONE, 16, 0);
  TcCtx tc;
  tc_setup(sh, tc);
  dep_release();
  const float* whf = reinterpret_cast<const float*>(sm + hb::WHF);
  float* dys = reinterpret_cast<float*>(sm + hb::DYS);
  uint8_t* XT = sm + hb::XT;
  uint8_t* H2 = sm + hb::H2;
  const int node = threadIdx.x & 127, half = threadIdx.x >> 7, f0 = half * 32;
  const uint32_t lb = lane_base(tc.tmem);
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const int64_t ntiles = (N + TILE - 1) / TILE;
  bool first = true, ok = true;
  for (int64_t tile = after_wait((int64_t)blockIdx.x); tile < ntiles; tile += gridDim.x) {
    const int64_t n = tile * TILE + node;
    const bool on = n < N;
    const int64_t nn = on ? n : N - 1;
    if (LBM_BWD_PF && threadIdx.x < NOUT + 8) {  // next tile: dy (10 FP32 planes), h2 (8 planes)
      const int64_t m0 = (tile + gridDim.x) * TILE;
      if (threadIdx.x < NOUT) l2_prefetch_nodes(dy, threadIdx.x, N, 4, m0, N);
      else l2_prefetch_nodes(h2, threadIdx.x - NOUT, N, 16, m0, N);
    }
    if (half == 0) {
      float d[NOUT];
#pragma unroll
      for (int o = 0; o < NOUT; ++o) {
        d[o] = on ? ld_prev(dy + o * N + nn) : 0.0f;
        dys[node * NOUT + o] = d[o];
      }
      st_col<NOUT>(XT, 128, 0, node, d);
    }
    copy_row<32, true>(H2, node, f0, h2, N, nn);
    __syncthreads();
    float dv[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) dv[c] = 0.0f;
#pragma unroll
    for (int o = 0; o < NOUT; ++o) {
      const float g = dys[node * NOUT + o];
#pragma unroll
      for (int c = 0; c < 32; ++c) dv[c] = fmaf(g, whf[o * HID + f0 + c], dv[c]);
    }
    if (on) st_pf32(dh, N, n, f0, dv);
    const bool acc = !first;
    if (!tc_run(sh, tc, stw, [&] {
          umma_nt(tc.tmem, smem_u32(XT), 16384, smem_u32(H2), 0, 64, 8, acc);
          umma_128xN(tc.tmem + 64, smem_u32(XT), 16384, smem_u32(sm + hb::ONE), 2048, 2, 16, acc);
        })) {
      ok = false;
      break;
    }
    first = false;
  }
  if (ok && (threadIdx.x >> 5) == 0) {
    float v[32], w[32], u[16];
    tmem_ld32(lb, v);
    tmem_ld32(lb + 32, w);
    tmem_ld16(lb + 64, u);
    const int o = threadIdx.x & 31;
    if (o < NOUT) {
      float* g = G + (int64_t)blockIdx.x * P::TRAINABLE;
      for (int i = 0; i < 32; ++i) {
        g[P::HEAD_W + o * HID + i] = v[i];
        g[P::HEAD_W + o * HID + 32 + i] = w[i];
      }
      g[P::HEAD_B + o] = u[0];
    }
  }
  if (!ok) zero_grad(G + (int64_t)blockIdx.x * P::TRAINABLE, P::HEAD_W, NOUT * HID + NOUT);
  tc_teardown(sh, tc);
}

// ---------------------------------------------------------------------------
// Round backward, part 1 (per node): recompute z_n = W_n [h; a] + b_n,
// dz_n = dh_out * GELU'(z_n), d[h; a] = dz_n W_n; accumulate dW_n (tensor
// cores, [h; a]^T dz_n) and db_n (sum of dz_n, in registers by a butterfly
// reduction over each warp's nodes).  Outputs dh_part = dh_out + d[h; a]_h
// and da = d[h; a]_a (FP32).
namespace rb1 {
// HA: [h; a] node-major (two SW128 blocks), A of the z_n recompute and, across
// its rows, of dW_n; DZ: dz node-major, A of d[h; a] and, across its rows, B of
// dW_n.  W_n [64 out x 128 in] read across its rows is B of d[h; a].
constexpr uint32_t HA = 0, DZ = 32768, WN = 49152, BN = 65536, DBR = 65792, SH = 66816,
                   BYTES = 66944;
}
#ifndef LBM_RB1_CTAS
#define LBM_RB1_CTAS 2  // resident CTAs per SM
#endif

template <bool EARLY>
__global__ void __launch_bounds__(256, LBM_RB1_CTAS) gnn_round_bwd1_kernel(
    const __nv_bfloat16* __restrict__ h_in, const __nv_bfloat16* __restrict__ a_in,
    const float* dh_out, float* __restrict__ dh_part, float* __restrict__ da,
    int round, float* __restrict__ G, Shape s, const uint8_t* __restrict__ packed, unsigned* stw) {
  if (!blob_ok(packed, stw)) return dep_sync();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = smem_align1024(smem_raw);
  TcShared* sh = reinterpret_cast<TcShared*>(sm + rb1::SH);
  const uint8_t* kr = packed + K::round_base(round);
  const bool mlp_only = variant_of(reinterpret_cast<const float*>(packed + K::NORM)) & VAR_MLP_ONLY;
  copy_g2s(sm + rb1::WN, kr + K::WN, 16384);
  copy_g2s(sm + rb1::BN, kr + K::BN, 256);
  __syncthreads();
  TcCtx tc;
  tc_setup(sh, tc);
  const float* bn = reinterpret_cast<const float*>(sm + rb1::BN);
  uint8_t* HA = sm + rb1::HA;
  uint8_t* DZ = sm + rb1::DZ;
  const int node = threadIdx.x & 127, half = threadIdx.x >> 7, f0 = half * 32;
  const uint32_t lb = lane_base(tc.tmem);
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const int64_t ntiles = (N + TILE - 1) / TILE;
  float dbacc = 0.0f;  // lane l: running sum of dz[f0 + l] over this warp's nodes
  bool first = true, ok = true;
  dep_sync();
  for (int64_t tile = EARLY ? after_wait((int64_t)blockIdx.x) : blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t n = tile * TILE + node;
    const bool on = n < N;
    const int64_t nn = on ? n : N - 1;
    if (LBM_BWD_PF && threadIdx.x < 32) {  // next tile: h, a (8 planes each), dh_out (16)
      const int64_t m0 = (tile + gridDim.x) * TILE;
      const int t = threadIdx.x;
      if (t < 8) l2_prefetch_nodes(h_in, t, N, 16, m0, N);
      else if (t < 16) l2_prefetch_nodes(a_in, t - 8, N, 16, m0, N);
      else l2_prefetch_nodes(dh_out, t - 16, N, 16, m0, N);
    }
    copy_row<32>(HA, node, f0, h_in, N, nn);
    copy_row<32>(HA + 16384, node, f0, a_in, N, nn);
    if (!tc_run(sh, tc, stw, [&] {
          umma_128xN(tc.tmem, smem_u32(HA), 16384, smem_u32(sm + rb1::WN), 8192, 2, 64, false);
        })) {
      ok = false;
      break;
    }
    {
      float dz[32], dho[32];
      tmem_ld32(lb + f0, dz);
      ld_pf32<EARLY>(dh_out, N, nn, f0, dho);
      act_and_grad(dz, bn + f0, 32, false, nullptr, dz);  // GELU'(z_n), packed pairs
#pragma unroll
      for (int c = 0; c < 32; ++c) dz[c] = (on && !mlp_only) ? dho[c] * dz[c] : 0.0f;
      st_row32(DZ, node, f0, dz);
      dbacc += warp_transpose_sum(dz);
    }
    const bool acc = !first;
    if (!tc_run(sh, tc, stw, [&] {
          umma_nt(tc.tmem, smem_u32(DZ), 0, smem_u32(sm + rb1::WN), 8192, 128, 4, false);
          umma_tt(tc.tmem + 128, smem_u32(HA), 16384, smem_u32(DZ), 0, 64, 8, acc);
        })) {
      ok = false;
      break;
    }
    first = false;
    {
      float d[32], dho[32];
      tmem_ld32(lb + f0, d);           // warp-collective: every lane takes part
      ld_pf32<EARLY>(dh_out, N, nn, f0, dho);  // again (an L2 hit): fewer values live across the MMA
#pragma unroll
      for (int c = 0; c < 32; ++c) d[c] += dho[c];
      if (on) st_pf32(dh_part, N, n, f0, d);
      tmem_ld32(lb + HID + f0, d);
      if (on) st_pf32(da, N, n, f0, d);
    }
    tc_fence_before();
    __syncthreads();
  }
  if (ok) {
    // D_wn[i][o] at columns 128..191 (row i = input feature of [h; a])
    const int row = 32 * ((threadIdx.x >> 5) & 3) + (threadIdx.x & 31);
    float* g = G + (int64_t)blockIdx.x * P::TRAINABLE + P::ROUND0 + round * P::ROUND_SIZE;
    float v[32];
    tmem_ld32(lb + 128 + f0, v);
    for (int c = 0; c < 32; ++c) g[P::NODE_W + (f0 + c) * 128 + row] = v[c];
    // db_n: the 4 warps of a feature half hold disjoint node sets; fixed order
    float* dbr = reinterpret_cast<float*>(sm + rb1::DBR);  // [8 warps][32]
    dbr[(threadIdx.x >> 5) * 32 + (threadIdx.x & 31)] = dbacc;
    __syncthreads();
    if (threadIdx.x < HID) {
      const int hh = threadIdx.x >> 5, l = threadIdx.x & 31;
      float t = 0.0f;
      for (int q = 0; q < 4; ++q) t += dbr[(hh * 4 + q) * 32 + l];
      g[P::NODE_B + threadIdx.x] = t;
    }
  } else {
    zero_grad(G + (int64_t)blockIdx.x * P::TRAINABLE + P::ROUND0 + round * P::ROUND_SIZE,
              P::NODE_W, P::ROUND_SIZE - P::NODE_W);
  }
  tc_teardown(sh, tc);
}

// ---------------------------------------------------------------------------
// Round backward, part 2 (pull form): for node j
//   dA_j = sum_k da_j * GELU'(A_j + B_{j+e_k} + c_k)
//   dB_j = sum_k da_i * GELU'(A_i + B_j + c_k),  i = j - e_k
//   dc_x,j / dc_y,j = the e_kx / e_ky weighted sums of the dA_j terms.
// dh_in = dh_part + [dA | dB] [W_a; W_b]; accumulates [dW_a; dW_b], db_e
// (= sum dA) on the tensor cores and the W_c columns (sum dc_x, sum dc_y) in
// registers (butterfly reduction over the warp's nodes).
namespace rb2 {
// DAB: [dA | dB] node-major, A of the dh product and, across its rows, of
// dW_a | dW_b; H: h node-major, B of the latter across its rows; ONE: 16 rows,
// row 0 ones
constexpr uint32_t DAB = 0, H = 32768, ONE = 49152, WABT = 53248, CK = 69632, CKH = 71680,
                   DCR = 72704, SH = 74752, BYTES = 74880;
}
// WALLS (the channel's graph): an edge whose far node lies beyond a wall
// (row outside [0, ny)) was left out of the forward's sum and passes no
// gradient; its neighbour address wraps to a row inside, so loads stay in
// range.
// Four threads per node, 16 features each: 16 warps of 128 registers per SM.
// Bound by the latency of the gathers and of the FP16 chains (FP16 pipe 47 %,
// issue 45 % with two threads per node at 233 registers: 8 warps); 64 x 256^2
// training step 11.18 -> 10.85 ms, a step of few tiles 37 -> 31 us per launch.
// dA and dB direction by direction in one loop (two independent chains)
// instead of one after the other: 10.85 -> 10.38 ms.
template <bool WALLS, bool EARLY>
__global__ void __launch_bounds__(512, 1) gnn_round_bwd2_kernel(
    const __half* __restrict__ ab, const float* da, const float* dh_part,
    const __nv_bfloat16* __restrict__ h_in,
    float* __restrict__ dh_in, int round, float* __restrict__ G, Shape s,
    const uint8_t* __restrict__ packed, unsigned* stw) {
  if (!blob_ok(packed, stw)) return dep_sync();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = smem_align1024(smem_raw);
  TcShared* sh = reinterpret_cast<TcShared*>(sm + rb2::SH);
  const uint8_t* kr = packed + K::round_base(round);
  zero_smem(sm + rb2::ONE, rb2::WABT - rb2::ONE);
  copy_g2s(sm + rb2::WABT, kr + K::WABT, 16384);
  copy_g2s(sm + rb2::CK, kr + K::CK, 2048);
  __syncthreads();
  ones_row(sm + rb2::ONE, 16, 0);
  {  // c_k as FP16 pairs
    const float* ckf = reinterpret_cast<const float*>(sm + rb2::CK);
    __half2* ckw = reinterpret_cast<__half2*>(sm + rb2::CKH);
    for (int i = threadIdx.x; i < 8 * HID / 2; i += blockDim.x)
      ckw[i] = __floats2half2_rn(ckf[2 * i], ckf[2 * i + 1]);
  }
  TcCtx tc;
  tc_setup(sh, tc);
  const __half2* ckh = reinterpret_cast<const __half2*>(sm + rb2::CKH);
  uint8_t* DAB = sm + rb2::DAB;
  uint8_t* H = sm + rb2::H;
  constexpr int NF = 16;  // features of a thread
  constexpr int GROUP = WALLS ? 1 : 2;  // directions whose loads are in flight together (more spill)
  float dcacc = 0.0f;  // lane l: running sum of value l of [dc_x | dc_y] over this warp's nodes
  const int node = threadIdx.x & 127, part = threadIdx.x >> 7, f0 = part * NF;
  const uint32_t lb = lane_base(tc.tmem);
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const int64_t ntiles = (N + TILE - 1) / TILE;
  bool first = true, ok = true;
  dep_sync();
  for (int64_t tile = EARLY ? after_wait((int64_t)blockIdx.x) : blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t n = tile * TILE + node;
    const bool on = n < N;
    const int64_t nn = on ? n : N - 1;
    const NodeXY p = node_xy(nn, s);
    const int c0 = f0, ch = c0 >> 3;
    // 2 GELU'(z) is evaluated in packed FP16 pairs (z = A + B + c_k is O(1)).
    // dA_j = da_j * sum_k GELU'(z_jk) factors: the sums over k (and their
    // e_kx / e_ky weighted forms) are taken in FP16 and multiplied by da_j
    // once.  dB_j needs the neighbours' da, so its terms are accumulated in
    // FP32 (gradients would underflow FP16).  Direction k of both sides goes
    // through together: two independent chains per pair of features.
    uint32_t aj[8], bj[8];
    {
      const uint4 a0 = __ldg(chunk8(ab, N, nn, c0)), a1 = __ldg(chunk8(ab, N, nn, c0 + 8));
      aj[0] = a0.x; aj[1] = a0.y; aj[2] = a0.z; aj[3] = a0.w;
      aj[4] = a1.x; aj[5] = a1.y; aj[6] = a1.z; aj[7] = a1.w;
      const uint4 b0 = __ldg(chunk8(ab, N, nn, HID + c0));
      const uint4 b1 = __ldg(chunk8(ab, N, nn, HID + c0 + 8));
      bj[0] = b0.x; bj[1] = b0.y; bj[2] = b0.z; bj[3] = b0.w;
      bj[4] = b1.x; bj[5] = b1.y; bj[6] = b1.z; bj[7] = b1.w;
    }
    __half2 S[8], Sx[8], Sy[8];  // sums over k of 2 GELU'(z_jk), e_kx and e_ky weighted
    float gB[16];
#pragma unroll
    for (int c = 0; c < 8; ++c) S[c] = Sx[c] = Sy[c] = __float2half2_rn(0.0f);
#pragma unroll
    for (int c = 0; c < 16; ++c) gB[c] = 0.0f;
#pragma unroll
    for (int g = 0; g < 8; g += GROUP) {  // directions k = g+1 .. g+GROUP
      uint4 bn[GROUP][2], ai[GROUP][2];
      float4 di[GROUP][4];
#pragma unroll
      for (int kk = 0; kk < GROUP; ++kk) {
        const int k = g + kk + 1;
        const int64_t j = checked(node_at(p, ex(k), ey(k), s), 0, N, stw);    // dA: B of j + e_k
        bn[kk][0] = __ldg(chunk8(ab, N, j, HID + c0));
        bn[kk][1] = __ldg(chunk8(ab, N, j, HID + c0 + 8));
        const int64_t i = checked(node_at(p, -ex(k), -ey(k), s), 0, N, stw);  // dB: A, da of j - e_k
        ai[kk][0] = __ldg(chunk8(ab, N, i, c0));
        ai[kk][1] = __ldg(chunk8(ab, N, i, c0 + 8));
#pragma unroll
        for (int t4 = 0; t4 < 4; ++t4) di[kk][t4] = ld_in<EARLY>(chunk4(da, N, i, c0 + 4 * t4));
      }
#pragma unroll
      for (int kk = 0; kk < GROUP; ++kk) {
        const int k = g + kk + 1;
        const __half2* c_k = ckh + (k - 1) * (HID / 2) + c0 / 2;
        const uint32_t* bw = reinterpret_cast<const uint32_t*>(bn[kk]);
        const uint32_t* aw = reinterpret_cast<const uint32_t*>(ai[kk]);
        const float* dv = reinterpret_cast<const float*>(di[kk]);
        // walls: the edges (j, k) and (j - e_k, k) exist if their far nodes lie inside
        const bool keep_a = !WALLS || (unsigned)(p.y + ey(k)) < (unsigned)s.ny;
        const bool keep_b = !WALLS || (unsigned)(p.y - ey(k)) < (unsigned)s.ny;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const __half2 z = __hadd2(__hadd2(u32_as_h2(aj[c]), c_k[c]), u32_as_h2(bw[c]));
          const __half2 gp = keep_a ? gelu_grad2_h2(z) : __float2half2_rn(0.0f);
          S[c] = __hadd2(S[c], gp);
          if (ex(k) > 0) Sx[c] = __hadd2(Sx[c], gp);
          if (ex(k) < 0) Sx[c] = __hsub2(Sx[c], gp);
          if (ey(k) > 0) Sy[c] = __hadd2(Sy[c], gp);
          if (ey(k) < 0) Sy[c] = __hsub2(Sy[c], gp);
          const __half2 w = __hadd2(__hadd2(u32_as_h2(aw[c]), c_k[c]), u32_as_h2(bj[c]));
          const float2 gq = keep_b ? __half22float2(gelu_grad2_h2(w)) : make_float2(0.0f, 0.0f);
          gB[2 * c] = fmaf(dv[2 * c], gq.x, gB[2 * c]);
          gB[2 * c + 1] = fmaf(dv[2 * c + 1], gq.y, gB[2 * c + 1]);
        }
      }
    }
    {
      float gA[16], v[32];  // v = [dc_x | dc_y] of this node
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 t = ld_in<EARLY>(chunk4(da, N, nn, c0 + 4 * i));
        const float dd[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {  // the factor 1/2 of 2 GELU' is applied here
          const int c = 4 * i + q;
          const float d = on ? 0.5f * dd[q] : 0.0f;
          const float2 sv = __half22float2(S[c >> 1]), sx = __half22float2(Sx[c >> 1]);
          const float2 sy = __half22float2(Sy[c >> 1]);
          gA[c] = d * ((c & 1) ? sv.y : sv.x);
          v[c] = d * ((c & 1) ? sx.y : sx.x);
          v[16 + c] = d * ((c & 1) ? sy.y : sy.x);
        }
      }
      *reinterpret_cast<uint4*>(DAB + node * 128 + ((ch ^ (node & 7)) << 4)) = pack_bf16x8(gA);
      *reinterpret_cast<uint4*>(DAB + node * 128 + (((ch + 1) ^ (node & 7)) << 4)) =
          pack_bf16x8(gA + 8);
      // dc sums over this warp's 32 nodes: lane l gets value l of [dc_x | dc_y]
      dcacc += warp_transpose_sum(v);
    }
#pragma unroll
    for (int c = 0; c < 16; ++c) gB[c] = on ? 0.5f * gB[c] : 0.0f;
    uint8_t* b1 = DAB + 16384;
    *reinterpret_cast<uint4*>(b1 + node * 128 + ((ch ^ (node & 7)) << 4)) = pack_bf16x8(gB);
    *reinterpret_cast<uint4*>(b1 + node * 128 + (((ch + 1) ^ (node & 7)) << 4)) =
        pack_bf16x8(gB + 8);
    copy_row<NF>(H, node, f0, h_in, N, nn);
    const bool acc = !first;
    if (!tc_run(sh, tc, stw, [&] {
          umma_128xN(tc.tmem, smem_u32(DAB), 16384, smem_u32(sm + rb2::WABT), 8192, 2, 64, false);
          umma_tt(tc.tmem + 64, smem_u32(DAB), 16384, smem_u32(H), 0, 64, 8, acc);
          umma_tn(tc.tmem + 128, smem_u32(DAB), 16384, smem_u32(sm + rb2::ONE), 2048, 16, 8, acc);
        })) {
      ok = false;
      break;
    }
    first = false;
    float d[NF], dp[NF];
    tmem_ld<NF>(lb + f0, d);
    if (on) {
      ld_pf<NF, EARLY>(dh_part, N, n, f0, dp);
#pragma unroll
      for (int c = 0; c < NF; ++c) d[c] += dp[c];
      st_pf<NF>(dh_in, N, n, f0, d);
    }
    tc_fence_before();
    __syncthreads();
  }
  if (ok) {
    const int row = 32 * ((threadIdx.x >> 5) & 3) + (threadIdx.x & 31);  // o' (a rows, then b rows)
    float* g = G + (int64_t)blockIdx.x * P::TRAINABLE + P::ROUND0 + round * P::ROUND_SIZE;
    const int o = row & 63;
    const int col_off = row < HID ? 0 : HID;
    float v[NF];
    tmem_ld<NF>(lb + 64 + f0, v);
    for (int c = 0; c < NF; ++c) g[P::EDGE_W + o * 130 + col_off + f0 + c] = v[c];
    if (part == 0) {
      float u[16];
      tmem_ld16(lb + 128, u);  // column sum of [dA | dB]
      if (row < HID) g[P::EDGE_B + o] = u[0];
    }
    // W_c columns: the 4 warps of a feature part hold disjoint node sets;
    // summed in fixed order.
    float* dcr = reinterpret_cast<float*>(sm + rb2::DCR);  // [16 warps][32]
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    dcr[w * 32 + lane] = dcacc;
    __syncthreads();
    if (threadIdx.x < 128) {
      const int pt = threadIdx.x >> 5, l = threadIdx.x & 31;
      float t = 0.0f;
      for (int q = 0; q < 4; ++q) t += dcr[(pt * 4 + q) * 32 + l];
      g[P::EDGE_W + (16 * pt + (l & 15)) * 130 + 128 + (l >> 4)] = t;
    }
  } else {
    zero_grad(G + (int64_t)blockIdx.x * P::TRAINABLE + P::ROUND0 + round * P::ROUND_SIZE,
              P::EDGE_W, P::NODE_W);
  }
  tc_teardown(sh, tc);
}

// ---------------------------------------------------------------------------
// Encoder backward: recompute x_hat, z1, g1, z2; dz2 = dh0 * GELU'(z2),
// dg1 = dz2 W2, dz1 = dg1 * GELU'(z1); accumulate
// D[o'][i'] = sum_n [dz2 | dz1][n][o'] [g1 | x_hat | 1][n][i'], which holds
// dW2, db2 (rows 0..63) and dW1, db1 (rows 64..127).  Optionally the input
// gradient dL/df_pre through x_hat (f_i, rho and u = j / rho).
namespace eb {
// Node-major tiles: G1 (A of the z2 product and, across its rows, B of dW2),
// DZ = [dz2 | dz1] (dz2: A of dg1; both, across their rows, A of the weight
// gradients); XH: 16 rows x_hat (12), ones (1), 0; DXH: the df partial sums.
// W2 read across its rows is B of dg1.
constexpr uint32_t G1 = 0, DZ = 16384, XH = 49152, W2 = 53248, W1F = 61440, B1 = 64512,
                   B2 = 64768, NORM = 65024, SH = 65152, DXH = 65280, BYTES = DXH + 12288;
}
#ifndef LBM_EB_CTAS
#define LBM_EB_CTAS 2  // resident CTAs per SM
#endif

// The channel's velocity feature is (sum f e + F/2)/rho with F = (fx, 0)
// (fxs[b] per lattice when set; fx = 0 and fxs NULL elsewhere); its
// derivative w.r.t. f_i is (e_i - u)/rho with that u.
template <bool EARLY>
__global__ void __launch_bounds__(256, LBM_EB_CTAS) gnn_encode_bwd_kernel(
    const float* __restrict__ f_pre, const float* dh0, float* __restrict__ df,
    float* __restrict__ G, Shape s, float fx, const float* __restrict__ fxs,
    const uint8_t* __restrict__ packed, unsigned* stw) {
  if (!blob_ok(packed, stw)) return dep_sync();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = smem_align1024(smem_raw);
  TcShared* sh = reinterpret_cast<TcShared*>(sm + eb::SH);
  zero_smem(sm + eb::XH, eb::W2 - eb::XH);
  copy_g2s(sm + eb::W2, packed + K::W2, 8192);
  copy_g2s(sm + eb::W1F, packed + K::W1F, 3712);
  __syncthreads();
  ones_row(sm + eb::XH, 16, NFEAT);
  // 1 / sigma (the forward encoder normalises by this product too), beside
  // the tensor-core context
  float* isg = reinterpret_cast<float*>(sm + eb::SH + 64);
  if (threadIdx.x < NFEAT)
    isg[threadIdx.x] = 1.0f / reinterpret_cast<const float*>(sm + eb::NORM)[NFEAT + threadIdx.x];
  TcCtx tc;
  tc_setup(sh, tc);
  const float* w1 = reinterpret_cast<const float*>(sm + eb::W1F);
  const float* b1 = reinterpret_cast<const float*>(sm + eb::B1);
  const float* b2 = reinterpret_cast<const float*>(sm + eb::B2);
  const float* nrm = reinterpret_cast<const float*>(sm + eb::NORM);
  float* dxh = reinterpret_cast<float*>(sm + eb::DXH);
  uint8_t* G1 = sm + eb::G1;
  uint8_t* DZ = sm + eb::DZ;
  uint8_t* XH = sm + eb::XH;
  const int node = threadIdx.x & 127, half = threadIdx.x >> 7, f0 = half * 32;
  const bool relu = variant_of(nrm) & VAR_MLP_ONLY;
  const uint32_t lb = lane_base(tc.tmem);
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const int64_t ntiles = (N + TILE - 1) / TILE;
  bool first = true, ok = true;
  dep_sync();
  for (int64_t tile = EARLY ? after_wait((int64_t)blockIdx.x) : blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t n = tile * TILE + node;
    const bool on = n < N;
    const int64_t nn = on ? n : N - 1;
    if (LBM_BWD_PF && threadIdx.x < Q + 16) {  // next tile: f_pre (9 FP32 planes), dh0 (16)
      const int64_t m0 = (tile + gridDim.x) * TILE;
      if (threadIdx.x < Q) l2_prefetch_nodes(f_pre, threadIdx.x, s.ps, 4, m0, N);
      else l2_prefetch_nodes(dh0, threadIdx.x - Q, N, 16, m0, N);
    }
    float fv[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) fv[q] = __ldg(f_pre + q * s.ps + nn);
    Moments m = moments9(fv);
    if (fxs || fx != 0.0f)
      m.ux += 0.5f * (fxs ? __ldg(fxs + nn / ((int64_t)s.nx * s.ny)) : fx) / m.rho;
    float xh[NFEAT];
#pragma unroll
    for (int q = 0; q < Q; ++q) xh[q] = (fv[q] - nrm[q]) * isg[q];
    xh[9] = (m.rho - nrm[9]) * isg[9];
    xh[10] = (m.ux - nrm[10]) * isg[10];
    xh[11] = (m.uy - nrm[11]) * isg[11];
    // GELU'(z1), the only later use of z1, kept as FP16 pairs (values in
    // [-0.2, 1.2]; dz1 is rounded to BF16 for the weight-gradient MMA anyway)
    __half2 gp1[16];
    {
      float z1[32], g[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        float z = b1[f0 + c];
#pragma unroll
        for (int j = 0; j < NFEAT; ++j) z = fmaf(w1[(f0 + c) * NFEAT + j], xh[j], z);
        z1[c] = z;
      }
      act_and_grad(z1, nullptr, 32, relu, g, z1);
#pragma unroll
      for (int c = 0; c < 16; ++c) gp1[c] = __floats2half2_rn(z1[2 * c], z1[2 * c + 1]);
      st_row32(G1, node, f0, g);
    }
    if (half == 0) st_col<NFEAT>(XH, 16, 0, node, xh);
    if (!tc_run(sh, tc, stw, [&] {
          umma_128xN(tc.tmem, smem_u32(G1), 0, smem_u32(sm + eb::W2), 0, 1, 64, false);
        })) {
      ok = false;
      break;
    }
    float d[32];
    {
      float z2[32], g0[32];
      tmem_ld32(lb + f0, z2);
      ld_pf32<EARLY>(dh0, N, nn, f0, g0);
      act_and_grad(z2, b2 + f0, 32, relu, nullptr, d);
#pragma unroll
      for (int c = 0; c < 32; ++c) d[c] = on ? g0[c] * d[c] : 0.0f;
    }
    st_row32(DZ, node, f0, d);
    if (!tc_run(sh, tc, stw, [&] {
          umma_nt(tc.tmem, smem_u32(DZ), 0, smem_u32(sm + eb::W2), 0, 64, 4, false);
        })) {
      ok = false;
      break;
    }
    tmem_ld32(lb + f0, d);
#pragma unroll
    for (int c = 0; c < 16; ++c) {  // dz1 = dg1 GELU'(z1) (0 for idle nodes)
      const float2 gp = __half22float2(gp1[c]);
      d[2 * c] *= gp.x;
      d[2 * c + 1] *= gp.y;
    }
    st_row32(DZ + 16384, node, f0, d);
    if (df) {
      float px[NFEAT];
#pragma unroll
      for (int j = 0; j < NFEAT; ++j) px[j] = 0.0f;
#pragma unroll
      for (int c = 0; c < 32; ++c) {
#pragma unroll
        for (int j = 0; j < NFEAT; ++j) px[j] = fmaf(d[c], w1[(f0 + c) * NFEAT + j], px[j]);
      }
#pragma unroll
      for (int j = 0; j < NFEAT; ++j) dxh[(half * 128 + node) * NFEAT + j] = px[j];
    }
    const bool acc = !first;
    if (!tc_run(sh, tc, stw, [&] {
          umma_tt(tc.tmem + 64, smem_u32(DZ), 16384, smem_u32(G1), 0, 64, 8, acc);
          umma_tn(tc.tmem + 128, smem_u32(DZ), 16384, smem_u32(XH), 2048, 16, 8, acc);
        })) {
      ok = false;
      break;
    }
    first = false;
    if (df && half == 0 && on) {
      float dx[NFEAT];
#pragma unroll
      for (int j = 0; j < NFEAT; ++j)
        dx[j] = (dxh[node * NFEAT + j] + dxh[(128 + node) * NFEAT + j]) * isg[j];
      const float ir = 1.0f / m.rho;
#pragma unroll
      for (int q = 0; q < Q; ++q)
        df[q * s.ps + n] =
            dx[q] + dx[9] + (dx[10] * (float(ex(q)) - m.ux) + dx[11] * (float(ey(q)) - m.uy)) * ir;
    }
    tc_fence_before();
    __syncthreads();
  }
  if (ok) {
    const int row = 32 * ((threadIdx.x >> 5) & 3) + (threadIdx.x & 31);
    float* g = G + (int64_t)blockIdx.x * P::TRAINABLE;
    float v[32];
    tmem_ld32(lb + 64 + f0, v);
    if (row < HID) {
      for (int c = 0; c < 32; ++c) g[P::ENC2_W + row * HID + f0 + c] = v[c];
    }
    if (half == 0) {
      float u[16];
      tmem_ld16(lb + 128, u);  // columns 64..79: x_hat (12), ones (1)
      if (row < HID) {
        g[P::ENC2_B + row] = u[12];
      } else {
        for (int j = 0; j < NFEAT; ++j) g[P::ENC1_W + (row - HID) * NFEAT + j] = u[j];
        g[P::ENC1_B + row - HID] = u[12];
      }
    }
  } else {
    zero_grad(G + (int64_t)blockIdx.x * P::TRAINABLE, 0, P::ROUND0);
  }
  tc_teardown(sh, tc);
}

// ---------------------------------------------------------------------------
// Sum of the per-CTA gradient rows, from the first to the last; every kernel
// writes its own parameters' columns in as many rows as it has CTAs.  A thread
// per parameter; bound by the latency of its loads, which are independent
// within batches of 32 rows (as many in flight as its 30 registers hold; 26 us
// for 512 rows before, most of them empty; 6 for 128 rows).
// accumulate: add to the gradient already in grad (the steps of a rollout).
struct GradRows {
  int enc, edge, node, head;
};
__global__ void __launch_bounds__(64) grad_reduce_kernel(const float* G, GradRows rows,
                                                         float* __restrict__ grad, bool accumulate,
                                                         const uint8_t* __restrict__ packed) {
  dep_sync();
  const int p = after_wait((int)(blockIdx.x * 64 + threadIdx.x));
  if (p >= P::TRAINABLE) return;
  int n = rows.enc;
  if (p >= P::HEAD_W)
    n = rows.head;
  else if (p >= P::ROUND0)
    n = (p - P::ROUND0) % P::ROUND_SIZE < P::NODE_W ? rows.edge : rows.node;
  // an invalid image: no kernel wrote its rows, the gradient is 0
  if (__ldg(reinterpret_cast<const unsigned*>(packed + K::MAGIC_SLOT)) != K::MAGIC) n = 0;
  constexpr int BATCH = 32;
  float acc = 0.0f;
  for (int r0 = 0; r0 < n; r0 += BATCH) {
    float v[BATCH];
#pragma unroll
    for (int i = 0; i < BATCH; ++i)
      v[i] = r0 + i < n ? ld_prev(G + (int64_t)(r0 + i) * P::TRAINABLE + p) : 0.0f;
#pragma unroll
    for (int i = 0; i < BATCH; ++i) acc += v[i];
  }
  grad[p] = accumulate ? grad[p] + acc : acc;
}

// AdamW (decoupled weight decay) on the trainable prefix.
__global__ void adamw_kernel(float* __restrict__ theta, const float* g,
                             float* __restrict__ m, float* __restrict__ v, float lr, float wd,
                             float b1, float b2, float eps, float bc1, float bc2) {
  dep_sync();
  const int p = after_wait((int)(blockIdx.x * blockDim.x + threadIdx.x));
  if (p >= P::TRAINABLE) return;
  const float gp = ld_prev(g + p);
  const float mp = b1 * m[p] + (1.0f - b1) * gp;
  const float vp = b2 * v[p] + (1.0f - b2) * gp * gp;
  m[p] = mp;
  v[p] = vp;
  const float mh = mp * bc1, vh = vp * bc2;
  theta[p] = theta[p] * (1.0f - lr * wd) - lr * mh / (sqrtf(vh) + eps);
}

// ---------------------------------------------------------------------------
// Launchers
cudaError_t launch_collide_loss(const float* f_pre, const float* y, const float* tgt,
                                const Shape& s, float tau, const float* taus,
                                const uint8_t* packed, double* lossp, int* nblk, float* dy,
                                float* f_pred, cudaStream_t st, const float* lw) {
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const unsigned blocks = (unsigned)((N + 255) / 256);
  *nblk = (int)blocks;
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  const bool early = tiles_alone(N);
  return launch_after(early, gnn_collide_loss_kernel<false>, blocks, 256, 0, st, f_pre, y, tgt, s, tau, taus,
                      0.0f, nullptr, packed, lossp, dy, f_pred, lw, stw);
}

cudaError_t launch_collide_loss_channel(const float* f_pre, const float* y, const float* tgt,
                                        const Shape& s, float tau, const float* taus, float gx,
                                        const float* gxs, const uint8_t* packed, double* lossp,
                                        int* nblk, float* dy, float* f_pred, cudaStream_t st,
                                        const float* lw) {
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const unsigned blocks = (unsigned)((N + 255) / 256);
  *nblk = (int)blocks;
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  const bool early = tiles_alone(N);
  return launch_after(early, gnn_collide_loss_kernel<true>, blocks, 256, 0, st, f_pre, y, tgt, s, tau, taus,
                      gx, gxs, packed, lossp, dy, f_pred, lw, stw);
}

cudaError_t launch_collide_adjoint(const float* f_pre, const float* y, const float* f_post,
                                   const float* tgt, const float* g_in, const Shape& s, float tau,
                                   const float* taus, const uint8_t* packed, float scale,
                                   float* dy, float* dfd, cudaStream_t st) {
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const bool early = tiles_alone(N);
  return launch_after(early, gnn_collide_adjoint_kernel, (unsigned)((N + 255) / 256), 256, 0, st, f_pre, y,
                      f_post, tgt, g_in, s, tau, taus, packed, scale, dy, dfd, stw);
}

cudaError_t launch_stream_adjoint_sum(const float* a, const float* b, float* out, const Shape& s,
                                      cudaStream_t st) {
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const bool early = tiles_alone(N);
  return launch_after(early, stream_adjoint_sum_kernel, (unsigned)((N + 255) / 256), 256, 0, st, a, b, out,
                      s, stw);
}

cudaError_t launch_loss_finish(const double* lossp, int nblk, double count, double* loss,
                               cudaStream_t st) {
  const bool early = nblk <= 512;
  return launch_after(early, loss_finish_kernel, 1, 1024, 0, st, lossp, nblk, count, loss);
}

static unsigned grad_grid(int64_t N, int per_sm) {
  unsigned g = grid_for(N, per_sm);
  return g > (unsigned)GRAD_ROWS ? (unsigned)GRAD_ROWS : g;
}

cudaError_t launch_gnn_backward(const BackwardLaunch& bl, const Shape& s, const uint8_t* packed,
                                cudaStream_t st) {
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  cudaError_t e;
  const bool early = tiles_alone(N);
  const GradRows rows{(int)grad_grid(N, LBM_EB_CTAS), (int)grad_grid(N, 1),
                      (int)grad_grid(N, LBM_RB1_CTAS), (int)grad_grid(N, LBM_HB_CTAS)};
  // head: dh2 -> dh[0]
  {
    const uint32_t bytes = hb::BYTES + 1024;
    if ((e = set_smem(gnn_head_bwd_kernel, bytes)) != cudaSuccess) return e;
    if ((e = launch_after(early, gnn_head_bwd_kernel, rows.head, 256, bytes, st, bl.dy, bl.h2, bl.dh[0],
                          bl.G, s, packed, stw)) != cudaSuccess)
      return e;
  }
  // rounds 2 and 1 (index 1, 0): dh[0] -> dh[1] (part) -> dh[0] (in)
  const __nv_bfloat16* hs[2] = {bl.h0, bl.h1};
  const __nv_bfloat16* as[2] = {bl.a0, bl.a1};
  const __half* abs_[2] = {bl.ab0, bl.ab1};
  for (int r = 1; r >= 0; --r) {
    {
      const uint32_t bytes = rb1::BYTES + 1024;
      auto* kern = early ? gnn_round_bwd1_kernel<true> : gnn_round_bwd1_kernel<false>;
      if ((e = set_smem(kern, bytes)) != cudaSuccess) return e;
      if ((e = launch_after(early, kern, rows.node, 256, bytes, st, hs[r], as[r], bl.dh[0],
                            bl.dh[1], bl.da, r, bl.G, s, packed, stw)) != cudaSuccess)
        return e;
    }
    {
      const uint32_t bytes = rb2::BYTES + 1024;
      auto* kern = bl.walls ? (early ? gnn_round_bwd2_kernel<true, true>
                                     : gnn_round_bwd2_kernel<true, false>)
                            : (early ? gnn_round_bwd2_kernel<false, true>
                                     : gnn_round_bwd2_kernel<false, false>);
      if ((e = set_smem(kern, bytes)) != cudaSuccess) return e;
      if ((e = launch_after(early, kern, rows.edge, 512, bytes, st, abs_[r], bl.da, bl.dh[1],
                            hs[r], bl.dh[0], r, bl.G, s, packed, stw)) != cudaSuccess)
        return e;
    }
  }
  {
    const uint32_t bytes = eb::BYTES + 1024;
    auto* kern = early ? gnn_encode_bwd_kernel<true> : gnn_encode_bwd_kernel<false>;
    if ((e = set_smem(kern, bytes)) != cudaSuccess) return e;
    if ((e = launch_after(early, kern, rows.enc, 256, bytes, st, bl.f_pre, bl.dh[0], bl.df,
                          bl.G, s, bl.fx, bl.fxs, packed, stw)) != cudaSuccess)
      return e;
  }
  return launch_after(early, grad_reduce_kernel, (P::TRAINABLE + 63) / 64, 64, 0, st, bl.G, rows, bl.grad,
                      bl.accumulate, packed);
}

cudaError_t launch_adamw(float* theta, const float* g, float* m, float* v, float lr, float wd,
                         float b1, float b2, float eps, float bc1, float bc2, cudaStream_t st) {
  return launch_after(true, adamw_kernel, (P::TRAINABLE + 255) / 256, 256, 0, st, theta, g, m, v, lr, wd,
                      b1, b2, eps, bc1, bc2);
}

}  // namespace lbmgnn
