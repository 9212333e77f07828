// GNN-enhanced collision, forward direction (paper Sec. 2.2-2.3, Eq. 3):
// parameter packing, the encoder kernel, and the message-passing round kernel
// (inner round, or last round fused with the head and either the Eq. 3
// collision + store or the raw head output).
//
// Work unit: a tile of 128 consecutive nodes (in the stacked-lattice node
// order).  A CTA of 256 threads owns one tile at a time (persistent loop over
// tiles); thread t handles node t % 128 and features 32*(t / 128) .. +32, so
// that warp w reads tensor-memory lanes 32*(w % 4).. of the accumulators.
// Dense layers are tcgen05 MMAs (M = 128 nodes, BF16 operands in 128-byte
// swizzled shared memory, FP32 accumulators in tensor memory).  Elementwise
// work (12->64 input layer, GELUs, the 8 messages per node) runs on the CUDA
// cores.  Between the kernels, h (BF16 [N][64]) and the per-node edge term
// B = W_b h (FP16 [N][64]) live in HBM; the 8 neighbour reads of B are served
// mostly from L2.  The node's own term A = W_a h is recomputed from h by the
// consuming round kernel (one 128x64x64 MMA per tile) instead of being stored.
// The training forward (gnn_forward) stores A | B ([N][128]) for the backward.
#include "gnn.cuh"
#include "gnn_launch.h"
#include "launch.h"

#ifndef LBM_PREFETCH
#define LBM_PREFETCH 1  // load the next tile's inputs while computing this one
#endif

namespace lbmgnn {

// ---------------------------------------------------------------------------
// Parameter packing: FP32 flat vector -> packed device image.
__device__ __forceinline__ void put_sw(uint8_t* blk, int row, int k, float v) {
  *reinterpret_cast<__nv_bfloat16*>(blk + sw128_off(row, k)) = __float2bfloat16_rn(v);
}

// The parameter vector: the kernel before (AdamW) may have written it.
struct PrevParams {
  const float* p;
  __device__ __forceinline__ float operator[](int i) const { return ld_prev(p + i); }
  __device__ __forceinline__ PrevParams operator+(int i) const { return {p + i}; }
};

__global__ void gnn_pack_kernel(const float* params, uint8_t* __restrict__ out, unsigned* stw) {
  dep_sync();
  const PrevParams p{after_wait(params)};
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  const int nth = gridDim.x * blockDim.x;
  float* w1f = reinterpret_cast<float*>(out + K::W1F);
  // the image's unused bytes
  for (int e = tid; e < 208; e += nth) reinterpret_cast<float*>(out + K::WHF)[NOUT * HID + e] = 0.0f;
  for (int e = tid; e < 256; e += nth)
    reinterpret_cast<float*>(out + K::round_base(e >> 7) + K::BN)[HID + (e & 127)] = 0.0f;
  for (int e = tid; e < HID * NFEAT; e += nth) w1f[e] = bf16_round(p[P::ENC1_W + e]);
  for (int e = tid; e < HID; e += nth) {
    reinterpret_cast<float*>(out + K::B1)[e] = p[P::ENC1_B + e];
    reinterpret_cast<float*>(out + K::B2)[e] = p[P::ENC2_B + e];
  }
  for (int e = tid; e < 31; e += nth)
    reinterpret_cast<float*>(out + K::NORM)[e] = e < 26 ? p[P::MU + e] : 0.0f;
  if (tid < 32) {  // the fixed values: finite mu, sigma > 0, s_df > 0, variant 0..7
    // (a lane each: one thread testing them one after the other took longer
    // than the rest of the pack, 10 us against 4)
    bool ok = true;
    if (tid < NFEAT) {
      const float mu = p[P::MU + tid], sg = p[P::SIGMA + tid];
      ok = isfinite(mu) && sg > 0.0f && isfinite(sg);
    } else if (tid == NFEAT) {
      ok = p[P::S_DF] > 0.0f && isfinite(p[P::S_DF]);
    } else if (tid == NFEAT + 1) {
      const float v = p[P::VARIANT];
      ok = v >= 0.0f && v <= (float)VAR_ALL && v == floorf(v);
    }
    ok = __all_sync(0xffffffffu, ok);
    if (tid == 0) {
      *reinterpret_cast<unsigned*>(out + K::MAGIC_SLOT) = ok ? K::MAGIC : 0u;
      if (!ok) atomicOr(stw, (unsigned)ST_BLOB);
    }
  }
  for (int e = tid; e < 16; e += nth)
    reinterpret_cast<float*>(out + K::BH)[e] = e < NOUT ? p[P::HEAD_B + e] : 0.0f;
  for (int e = tid; e < NOUT * HID; e += nth)
    reinterpret_cast<float*>(out + K::WHF)[e] = bf16_round(p[P::HEAD_W + e]);
  // the 4,096-element blocks go to threads of their own (64 blocks of 256: a
  // thread then walks through one of them, not through all)
  auto at = [&](int section) { return (tid + nth - section * HID * HID % nth) % nth; };
  for (int e = at(1); e < HID * HID; e += nth) {
    const int o = e / HID, i = e % HID;
    const float w = p[P::ENC2_W + o * HID + i];
    put_sw(out + K::W2, o, i, w);
    put_sw(out + K::W2T, i, o, w);
  }
  for (int e = tid; e < 16 * HID; e += nth) {
    const int o = e / HID, i = e % HID;
    put_sw(out + K::WH, o, i, o < NOUT ? p[P::HEAD_W + o * HID + i] : 0.0f);
  }
  for (int e = at(2); e < HID * HID; e += nth) {
    const int o = e / HID, k = e % HID;
    const int j = k < 16 ? k : k - 16;
    const float w = (k < 32 && j < NFEAT) ? p[P::ENC1_W + o * NFEAT + j] : 0.0f;
    put_sw(out + K::W1X, o, k, w);
  }
  for (int r = 0; r < 2; ++r) {
    const PrevParams pr = p + P::ROUND0 + r * P::ROUND_SIZE;
    uint8_t* kr = out + K::round_base(r);
    const PrevParams we = pr + P::EDGE_W;  // [64][130]
    const PrevParams wn = pr + P::NODE_W;  // [64][128]
    for (int e = at(3 + r); e < HID * HID; e += nth) {
      const int o = e / HID, i = e % HID;
      const float wa = we[o * 130 + i], wb = we[o * 130 + HID + i];
      put_sw(kr + K::WAB, o, i, wa);
      put_sw(kr + K::WAB, HID + o, i, wb);
      put_sw(kr + K::WABT, i, o, wa);
      put_sw(kr + K::WABT + 8192, i, o, wb);
      const float nh = wn[o * 128 + i], na = wn[o * 128 + HID + i];
      put_sw(kr + K::WN, o, i, nh);
      put_sw(kr + K::WN + 8192, o, i, na);
      put_sw(kr + K::WNT, i, o, nh);
      put_sw(kr + K::WNT, HID + i, o, na);
    }
    for (int e = tid; e < 8 * HID; e += nth) {
      const int k = e / HID + 1, o = e % HID;
      const float wcx = bf16_round(we[o * 130 + 128]), wcy = bf16_round(we[o * 130 + 129]);
      reinterpret_cast<float*>(kr + K::CK)[e] =
          (float(ex(k)) * wcx + float(ey(k)) * wcy) + pr[P::EDGE_B + o];
    }
    for (int e = tid; e < HID; e += nth) {
      reinterpret_cast<float*>(kr + K::BE)[e] = pr[P::EDGE_B + e];
      reinterpret_cast<float*>(kr + K::BN)[e] = pr[P::NODE_B + e];
    }
  }
}

// ---------------------------------------------------------------------------
// Encoder: pre-collision populations -> h0 (BF16) and the round-0 edge terms.
// Layer 1 (12 -> 64) runs on the tensor cores on [x_hi | x_lo] (see K::W1X),
// layer 2 and the round-0 edge terms A | B as BF16 MMAs; 128 TMEM columns are
// reused by the three products, so up to 3 CTAs share an SM.
namespace enc {
constexpr uint32_t W1X = 0, W2 = 8192, WAB = 16384, X1 = 32768, X = 49152, B1 = 65536,
                   B2 = 65792, NORM = 66048, SH = 66176, BYTES = 66304;
}

#ifndef LBM_ENC_CTAS
#define LBM_ENC_CTAS 2  // resident encoder CTAs per SM
#endif
// (The training forward's encoder; an inference step has that of gnn_mlp.cu.)
template <class Geo>
__global__ void __launch_bounds__(256, LBM_ENC_CTAS) gnn_encode_kernel(
    const float* __restrict__ f, Geo geo, const uint8_t* __restrict__ packed,
    __nv_bfloat16* __restrict__ h0_out, __half* __restrict__ ab_out, unsigned* stw) {
  if (!blob_ok(packed, stw)) return dep_sync();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = smem_align1024(smem_raw);
  TcShared* sh = reinterpret_cast<TcShared*>(sm + enc::SH);
  copy_g2s(sm + enc::W1X, packed + K::W1X, 8192);
  copy_g2s(sm + enc::W2, packed + K::W2, 8192);
  copy_g2s(sm + enc::WAB, packed + K::round_base(0) + K::WAB, 16384);
  copy_g2s(sm + enc::B1, packed + K::B1, 256 + 256 + 128);  // B1, B2, NORM
  __syncthreads();
  if (threadIdx.x < NFEAT) {  // sigma -> 1/sigma
    float* nrm = reinterpret_cast<float*>(sm + enc::NORM);
    nrm[NFEAT + threadIdx.x] = 1.0f / nrm[NFEAT + threadIdx.x];
  }
  TcCtx tc;
  tc_setup(sh, tc, 128);
  const float* b1 = reinterpret_cast<const float*>(sm + enc::B1);
  const float* b2 = reinterpret_cast<const float*>(sm + enc::B2);
  const float* nrm = reinterpret_cast<const float*>(sm + enc::NORM);
  uint8_t* X1 = sm + enc::X1;
  uint8_t* X = sm + enc::X;
  const int node = threadIdx.x & 127, half = threadIdx.x >> 7, f0 = half * 32;
  const uint32_t lb = lane_base(tc.tmem);
  const int64_t N = geo.count();
  const int64_t base = geo.base(), ps = geo.ps();
  const int64_t ntiles = (N + TILE - 1) / TILE;
  const bool relu = variant_of(nrm) & VAR_MLP_ONLY;

  // populations of node `t * TILE + node` of tile t
  auto load_f = [&](int64_t t, float (&v)[Q]) {
    const int64_t m = t * TILE + node;
    const int64_t mm = m < N ? m : N - 1;
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = __ldg(f + q * ps + base + mm);
  };
  float fnext[Q];
  dep_sync();
  if (blockIdx.x < ntiles) load_f(blockIdx.x, fnext);

  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t n = tile * TILE + node;
    const bool on = n < N;
    {
      float fv[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) fv[q] = fnext[q];
#if LBM_PREFETCH
      // the next tile's loads are in flight while this tile is computed
      if (tile + gridDim.x < ntiles) load_f(tile + gridDim.x, fnext);
#endif
      const Moments m = moments9(fv);
      float xh[16];
#pragma unroll
      for (int q = 0; q < Q; ++q) xh[q] = (fv[q] - nrm[q]) * nrm[NFEAT + q];
      xh[9] = (m.rho - nrm[9]) * nrm[NFEAT + 9];
      // channel: the force-corrected velocity (sum f e + F/2) / rho
      float ux = m.ux;
      if constexpr (Geo::kWalls) ux += 0.5f * geo.force_x(geo.pos(base + (n < N ? n : N - 1))) / m.rho;
      xh[10] = (ux - nrm[10]) * nrm[NFEAT + 10];
      xh[11] = (m.uy - nrm[11]) * nrm[NFEAT + 11];
      xh[12] = xh[13] = xh[14] = xh[15] = 0.0f;
      // half 0 writes x_hi (k 0..15), half 1 writes x_lo = x - x_hi (k 16..31)
      float v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float hi = bf16_round(xh[j]);
        v[j] = half == 0 ? hi : xh[j] - hi;
      }
      const int ch = half * 2;
      *reinterpret_cast<uint4*>(X1 + node * 128 + ((ch ^ (node & 7)) << 4)) = pack_bf16x8(v);
      *reinterpret_cast<uint4*>(X1 + node * 128 + (((ch + 1) ^ (node & 7)) << 4)) =
          pack_bf16x8(v + 8);
    }
    if (!tc_run(sh, tc, stw, [&] {
          umma_128xN(tc.tmem, smem_u32(X1), 0, smem_u32(sm + enc::W1X), 0, 1, 64, false, 2);
        }))
      break;
    float g[32];
    tmem_ld32(lb + f0, g);
    bias_act(g, b1 + f0, 32, relu);
    st_row32(X, node, f0, g);
    if (!tc_run(sh, tc, stw, [&] {
          umma_128xN(tc.tmem, smem_u32(X), 0, smem_u32(sm + enc::W2), 0, 1, 64, false);
        }))
      break;
    tmem_ld32(lb + f0, g);
    bias_act(g, b2 + f0, 32, relu);
    if (on && h0_out) st_pb32(h0_out, N, n, f0, g);
    st_row32(X, node, f0, g);  // the MMA that read X has completed
    // A | B = h0 [W_a; W_b]^T ([N][128])
    if (!tc_run(sh, tc, stw, [&] {
          umma_128xN(tc.tmem, smem_u32(X), 0, smem_u32(sm + enc::WAB), 0, 1, 128, false);
        }))
      break;
    tmem_ld32(lb + f0, g);
    if (on) st_ph32(ab_out, N, n, f0, g);
    tmem_ld32(lb + HID + f0, g);
    if (on) st_ph32(ab_out, N, n, HID + f0, g);
#if !LBM_PREFETCH
    if (tile + gridDim.x < ntiles) load_f(tile + gridDim.x, fnext);
#endif
    tc_fence_before();
    __syncthreads();
  }
  tc_teardown(sh, tc, 128);
}

// ---------------------------------------------------------------------------
// Message-passing round r.  MODE 0: inner round -> h_out, AB of round r+1.
// MODE 1: last round + head + Eq. 3 collision -> f_out (pull from f_post).
// MODE 2: last round + head -> y [10][N] (FP32) and h_out = h2.
// Shared-memory layout of a CTA of NG groups: per group g its node-state tile
// H (16 KB) and aggregated-message tile Ag (16 KB) at g * 32 KB, then the
// weights shared by the groups.  With A recomputed from h (AH), WX holds only
// the next round's W_b (8 KB) or the head, and this round's W_a sits at WA.
template <int NG>
struct RndL {
  static constexpr uint32_t WN = NG * 32768, WX = WN + 16384, WA = WX + 8192, CK = WX + 16384,
                            BN = CK + 2048, BH = BN + 256, NORM = BH + 64, CKH = NORM + 128,
                            SH = CKH + 1024, BYTES = SH + 64;
};

struct RoundArgs {
  const __nv_bfloat16* h_in;   // [N][64]
  const __half* ab_in;         // [N][128] FP16: A = W_a h, B = W_b h of this round, or
                               // [N][64] B alone (A recomputed from h_in)
  __nv_bfloat16* h_out;        // [N][64] (MODE 0, 2) or NULL
  __nv_bfloat16* a_out;        // [N][64] aggregated messages (saved for training) or NULL
  __half* ab_out;              // next round's A | B or B alone (MODE 0), FP16
  float* y_out;                // [10][N] (MODE 2)
  const float* f_post;         // stored state to pull from (MODE 1)
  float* f_out;                // MODE 1
  float tau;
  const float* taus;           // per-lattice tau or NULL
  int round;
  // Inference path: h0.  For the MLP-only network (no message passing) the
  // inner round then returns at once and the last round reads h0 from here.
  const __nv_bfloat16* h_skip;
};

#ifndef LBM_ROUND_CTAS
#define LBM_ROUND_CTAS 2
#endif
#ifndef LBM_ROUND_TPN
#define LBM_ROUND_TPN 1  // threads per node of the round kernel (1, 2 or 4)
#endif
#ifndef LBM_ROUND_GROUPS
#define LBM_ROUND_GROUPS 2  // independent tile groups per CTA
#endif
#ifndef LBM_NBR_GROUP
#define LBM_NBR_GROUP 4  // neighbour loads in flight per thread and chunk
#endif
// A CTA runs NG groups of 128 TPN threads; each group works through its own
// sequence of tiles with its own operands, mbarrier and 128 tensor-memory
// columns.  In a group, TPN threads per node each own FPT = 64 / TPN
// features; warp w reads tensor-memory lanes 32 (w % 4)..  AH: the edge
// terms come as B alone and A = W_a h is computed here from h.
template <int TPN>
constexpr int round_ctas() {  // resident CTAs per SM
  return TPN == 4 ? 1 : LBM_ROUND_CTAS;
}
template <int MODE, int TPN, int NG, bool AH, class Geo>
__global__ void __launch_bounds__(128 * TPN * NG, round_ctas<TPN>()) gnn_round_kernel(
    RoundArgs ra, Geo geo, const uint8_t* __restrict__ packed, unsigned* stw) {
  if (!blob_ok(packed, stw)) return dep_sync();
  if ((MODE == 0 || MODE == 1) && ra.h_skip &&
      (variant_of(reinterpret_cast<const float*>(packed + K::NORM)) & VAR_MLP_ONLY))
    return dep_sync();  // MLP-only network: no rounds; its inference step is the fused kernel (gnn_mlp.cu)
  constexpr int FPT = HID / TPN;
  constexpr int SL = FPT < 32 ? FPT : 32;  // feature slice of the epilogues
  constexpr int GT = 128 * TPN;            // threads per group
  using L = RndL<NG>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = smem_align1024(smem_raw);
  TcShared* sh = reinterpret_cast<TcShared*>(sm + L::SH);
  const uint8_t* kr = packed + K::round_base(ra.round);
  copy_g2s(sm + L::WN, kr + K::WN, 16384);
  if (AH) copy_g2s(sm + L::WA, kr + K::WAB, 8192);
  if (MODE == 0 && AH)  // rows 64..127 of the next round's W_ab block: W_b
    copy_g2s(sm + L::WX, packed + K::round_base(ra.round + 1) + K::WAB + 8192, 8192);
  else if (MODE == 0)
    copy_g2s(sm + L::WX, packed + K::round_base(ra.round + 1) + K::WAB, 16384);
  else
    copy_g2s(sm + L::WX, packed + K::WH, 2048);
  copy_g2s(sm + L::CK, kr + K::CK, 2048);
  copy_g2s(sm + L::BN, kr + K::BN, 256);
  copy_g2s(sm + L::BH, packed + K::BH, 64);
  copy_g2s(sm + L::NORM, packed + K::NORM, 128);
  __syncthreads();
  {  // c_k as FP16 pairs
    const float* ckf = reinterpret_cast<const float*>(sm + L::CK);
    __half2* ckw = reinterpret_cast<__half2*>(sm + L::CKH);
    for (int i = threadIdx.x; i < 8 * HID / 2; i += blockDim.x)
      ckw[i] = __floats2half2_rn(ckf[2 * i], ckf[2 * i + 1]);
  }
  const int grp = threadIdx.x / GT, tg = threadIdx.x % GT;
  TcCtx tc;
  tc_setup_groups(sh, tc, NG, grp, 128);
  const __half2* ckh = reinterpret_cast<const __half2*>(sm + L::CKH);
  const float* bn = reinterpret_cast<const float*>(sm + L::BN);
  const float* bh = reinterpret_cast<const float*>(sm + L::BH);
  const float* nrm = reinterpret_cast<const float*>(sm + L::NORM);
  uint8_t* H = sm + grp * 32768;
  uint8_t* Ag = H + 16384;
  const int node = tg & 127, part = tg >> 7, f0 = part * FPT;
  const uint32_t lb = lane_base(tc.tmem);
  const int64_t N = geo.count();
  const int64_t base = geo.base(), ps = geo.ps();
  const int64_t ntiles = (N + TILE - 1) / TILE;
  const int64_t stride = (int64_t)gridDim.x * NG;
  int64_t first = (int64_t)blockIdx.x * NG + grp;
  const int variant = variant_of(nrm);
  const bool mlp_only = variant & VAR_MLP_ONLY;
  const __nv_bfloat16* h_src = (mlp_only && ra.h_skip) ? ra.h_skip : ra.h_in;
  volatile int* abort_word = &sh[grp].abort;
  auto run = [&](auto issue) {
    tc_run_group_flag(tc, abort_word, grp, GT, issue);
    return true;
  };

  // The inputs are the kernel before's outputs; with four threads per node this
  // one is launched early (round_launch).
  constexpr bool EARLY = TPN == 4;
  // raw BF16 h (features f0.. of node `t * TILE + node`) of tile t
  uint4 hnext[FPT / 8];
  auto load_h = [&](int64_t t) {
    const int64_t m = t * TILE + node;
    const int64_t mm = m < N ? m : N - 1;
#pragma unroll
    for (int c = 0; c < FPT / 8; ++c) hnext[c] = ld_in<EARLY>(chunk8(h_src, N, mm, f0 + 8 * c));
  };
  dep_sync();
  if constexpr (EARLY) first = after_wait(first);
  if (AH && first < ntiles) load_h(first);

  for (int64_t tile = first; tile < ntiles; tile += stride) {
    const int64_t n = tile * TILE + node;
    const bool on = n < N;
    const int64_t nn = on ? n : N - 1;
    const GeoPos p = geo.pos(base + nn);
    if constexpr (AH) {  // h -> shared memory, A = h W_a^T -> tensor memory columns 0..63
#pragma unroll
      for (int c = 0; c < FPT / 8; ++c) {  // the BF16 words go to the swizzled row as they are
        const int chunk = (f0 >> 3) + c;
        *reinterpret_cast<uint4*>(H + node * 128 + ((chunk ^ (node & 7)) << 4)) = hnext[c];
      }
      if (LBM_PREFETCH && tile + stride < ntiles) load_h(tile + stride);
      if (!mlp_only && !run([&] {
            umma_128xN(tc.tmem, smem_u32(H), 0, smem_u32(sm + L::WA), 0, 1, 64, false);
          }))
        break;
    } else {  // h -> shared memory
#pragma unroll
      for (int s0 = 0; s0 < FPT; s0 += SL) {
        float h[SL];
#pragma unroll
        for (int c = 0; c < SL / 8; ++c)
          unpack_bf16x8(ld_in<EARLY>(chunk8(h_src, N, nn, f0 + s0 + 8 * c)), h + 8 * c);
        st_row<SL>(H, node, f0 + s0, h);
      }
    }
    if (mlp_only) {  // no message passing: a = 0, h unchanged
      if (on && ra.a_out) {
        const float zero[SL] = {};
#pragma unroll
        for (int s0 = 0; s0 < FPT; s0 += SL) st_pb<SL>(ra.a_out, N, n, f0 + s0, zero);
      }
    } else {
    // messages m_ik = GELU(A_i + B_j + c_k), summed over the 8 neighbours, in
    // packed FP16 pairs; per 16-feature chunk the neighbour loads are issued
    // LBM_NBR_GROUP at a time.
#pragma unroll
    for (int sc = 0; sc < FPT / 16; ++sc) {
      const int c0 = f0 + 16 * sc;
      uint32_t aw[8];
      if constexpr (AH) {
        float av[16];
        tmem_ld16(lb + c0, av);
#pragma unroll
        for (int c = 0; c < 8; ++c) aw[c] = h2_as_u32(__floats2half2_rn(av[2 * c], av[2 * c + 1]));
      } else {
        const uint4 a0 = ld_in<EARLY>(chunk8(ra.ab_in, N, nn, c0));
        const uint4 a1 = ld_in<EARLY>(chunk8(ra.ab_in, N, nn, c0 + 8));
        aw[0] = a0.x, aw[1] = a0.y, aw[2] = a0.z, aw[3] = a0.w;
        aw[4] = a1.x, aw[5] = a1.y, aw[6] = a1.z, aw[7] = a1.w;
      }
      // Each message 2 GELU(z) = z + z tanh(u) is formed by one fused
      // operation (exactly 0 once tanh(u) saturates at -1, however large |z|)
      // and then added to the sum; the 1/2 is applied once to the sum.
      __half2 acc[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[c] = __float2half2_rn(0.0f);
#pragma unroll
      for (int g = 0; g < 8; g += LBM_NBR_GROUP) {  // neighbours g .. g+LBM_NBR_GROUP-1
        uint4 braw[LBM_NBR_GROUP][2];
#pragma unroll
        for (int k = 0; k < LBM_NBR_GROUP; ++k) {
          const int64_t j = checked(geo_nbr(p, ex(g + k + 1), ey(g + k + 1)) - base, 0, N, stw);
          constexpr int BOFF = AH ? 0 : HID;  // B's first feature in ab_in
          braw[k][0] = ld_in<EARLY>(chunk8(ra.ab_in, N, j, BOFF + c0));
          braw[k][1] = ld_in<EARLY>(chunk8(ra.ab_in, N, j, BOFF + c0 + 8));
        }
#pragma unroll
        for (int k = 0; k < LBM_NBR_GROUP; ++k) {
          const uint32_t* bw = reinterpret_cast<const uint32_t*>(braw[k]);
          const __half2* c_k = ckh + (g + k) * (HID / 2) + c0 / 2;
          const __half2 c0h = __float2half2_rn(0.7978845608028654f);
          const __half2 c1h = __float2half2_rn(0.0356774081363001f);
          // channel: no message from a neighbour beyond a wall (its address
          // wrapped to a row inside, so the load stays in range)
          const __half2 keep = __float2half2_rn(geo.inside(p, ey(g + k + 1)) ? 1.0f : 0.0f);
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const __half2 z = __hadd2(__hadd2(u32_as_h2(aw[c]), c_k[c]), u32_as_h2(bw[c]));
            const __half2 u = __hmul2(z, __hfma2(c1h, __hmul2(z, z), c0h));
            if constexpr (Geo::kWalls)
              acc[c] = __hadd2(acc[c], __hmul2(keep, __hfma2(z, tanh_h2(u), z)));
            else
              acc[c] = __hadd2(acc[c], __hfma2(z, tanh_h2(u), z));
          }
        }
      }
      float av[16];
      const __half2 half_h2 = __float2half2_rn(0.5f);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const float2 t = __half22float2(__hmul2(acc[c], half_h2));
        av[2 * c] = t.x;
        av[2 * c + 1] = t.y;
      }
      const int ch = c0 >> 3;
      *reinterpret_cast<uint4*>(Ag + node * 128 + ((ch ^ (node & 7)) << 4)) = pack_bf16x8(av);
      *reinterpret_cast<uint4*>(Ag + node * 128 + (((ch + 1) ^ (node & 7)) << 4)) =
          pack_bf16x8(av + 8);
      if (on && ra.a_out) {
        *chunk8w(ra.a_out, N, n, c0) = pack_bf16x8(av);
        *chunk8w(ra.a_out, N, n, c0 + 8) = pack_bf16x8(av + 8);
      }
    }
    // node update: h <- h + GELU(W_n [h; a] + b_n)
    if (!run([&] {
          umma_128xN(tc.tmem, smem_u32(H), 16384, smem_u32(sm + L::WN), 8192, 2, 64, false);
        }))
      break;
    }
    // new h (the node-update MMA has completed: H may be overwritten)
#pragma unroll
    for (int s0 = 0; s0 < FPT; s0 += SL) {
      float h[SL];
      ld_row<SL>(H, node, f0 + s0, h);  // h as stored (BF16)
      if (!mlp_only) {
        float z[SL];
        tmem_ld<SL>(lb + f0 + s0, z);
#pragma unroll
        for (int c = 0; c < SL; c += 2) {
          const float2 g = gelu2(__fadd2_rn(make_float2(z[c], z[c + 1]),
                                            make_float2(bn[f0 + s0 + c], bn[f0 + s0 + c + 1])));
          const float2 hn = __fadd2_rn(make_float2(h[c], h[c + 1]), g);
          h[c] = hn.x;
          h[c + 1] = hn.y;
        }
      }
      if (on && ra.h_out) st_pb<SL>(ra.h_out, N, n, f0 + s0, h);
      st_row<SL>(H, node, f0 + s0, h);
    }
    if (MODE == 0) {  // next round's A | B, or B alone
      if (!run([&] {
            umma_128xN(tc.tmem, smem_u32(H), 0, smem_u32(sm + L::WX), 0, 1, AH ? 64 : 128, false);
          }))
        break;
#pragma unroll
      for (int s0 = 0; s0 < FPT; s0 += SL) {
        float a[SL];
        tmem_ld<SL>(lb + f0 + s0, a);
        if (on) st_ph<SL>(ra.ab_out, N, n, f0 + s0, a);
        if constexpr (!AH) {
          tmem_ld<SL>(lb + HID + f0 + s0, a);
          if (on) st_ph<SL>(ra.ab_out, N, n, HID + f0 + s0, a);
        }
      }
    } else {
      if (!run([&] {
            umma_128xN(tc.tmem, smem_u32(H), 0, smem_u32(sm + L::WX), 0, 1, 16, false);
          }))
        break;
      if (part == 0) {
        float y[16];
        tmem_ld16(lb, y);
#pragma unroll
        for (int o = 0; o < NOUT; ++o) y[o] += bh[o];
        if (MODE == 2) {
          if (on) {
#pragma unroll
            for (int o = 0; o < NOUT; ++o) ra.y_out[(int64_t)o * N + n] = y[o];
          }
        } else {
          // Eq. 3 on the pre-collision populations pulled from the stored state
          float fv[Q];
#pragma unroll
          for (int q = 0; q < Q; ++q)
            fv[q] = __ldg(ra.f_post + q * ps +
                          checked(geo_nbr(p, -ex(q), -ey(q)), base, base + N, stw));
          const Moments mm = moments9(fv);
          const float usq15 = 1.5f * (mm.ux * mm.ux + mm.uy * mm.uy);
          const float tau = geo.tau(p, ra.tau, ra.taus);
          const float tadj = tau_adj_of(y[0], variant);
          const float inv = 1.0f / (tau * tadj);
          const float sdf = nrm[24];
          float d[Q];
#pragma unroll
          for (int q = 0; q < Q; ++q) d[q] = sdf * y[1 + q];
          if (variant & VAR_CONSERVATIVE) conserve9(d);
          if (on) {
#pragma unroll
            for (int q = 0; q < Q; ++q) {
              const float fe = feq_i(q, mm, usq15);
              ra.f_out[q * ps + base + n] = fv[q] - (fv[q] - fe) * inv + d[q];
            }
          }
        }
      }
    }
    if (AH && !LBM_PREFETCH && tile + stride < ntiles) load_h(tile + stride);
    tc_fence_before();
    group_sync(grp, GT);
    if (*abort_word) {  // a tensor-core wait gave up: the group stops here
      if (tg == 0) raise_status(stw, ST_TIMEOUT);
      break;
    }
  }
  tc_teardown_groups(sh, NG, 128);
}

// ---------------------------------------------------------------------------
// Launchers
cudaError_t launch_gnn_pack(const float* params, uint8_t* packed, cudaStream_t st) {
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  return launch_after(true, gnn_pack_kernel, 64, 256, 0, st, params, packed, stw);
}


template <class Geo>
static cudaError_t encode_t(const float* f, const Geo& geo, int64_t N, const uint8_t* packed,
                            __nv_bfloat16* h0, __half* ab, cudaStream_t st) {
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  const uint32_t bytes = enc::BYTES + 1024;
  cudaError_t e;
  if ((e = set_smem(gnn_encode_kernel<Geo>, bytes)) != cudaSuccess) return e;
  gnn_encode_kernel<Geo><<<grid_for(N, LBM_ENC_CTAS), 256, bytes, st>>>(f, geo, packed, h0, ab, stw);
  return cudaGetLastError();
}

template <int MODE, int T, int G, bool AH, class Geo>
static cudaError_t round_launch(const RoundArgs& ra, const Geo& geo, unsigned grid,
                                const uint8_t* packed, unsigned* stw, cudaStream_t st) {
  const uint32_t bytes = RndL<G>::BYTES + 1024;
  cudaError_t e;
  if ((e = set_smem(gnn_round_kernel<MODE, T, G, AH, Geo>, bytes)) != cudaSuccess) return e;
  return launch_after(T == 4, gnn_round_kernel<MODE, T, G, AH, Geo>, grid, 128 * T * G, bytes, st, ra, geo,
                      packed, stw);
}

// Threads per node and tiles per CTA by the tiles that an SM gets (whole step
// of 128 x n lattices, 152 SMs).  One tile: the kernel takes as long as that
// tile, which four threads per node shorten.  Otherwise one thread per node and
// four tiles at a time have the higher rate, but an SM then takes its tiles in
// pairs (a CTA of two groups), so that an odd number costs as much as the next
// even one; two threads per node and two tiles at a time take them singly:
// 50 us against 60 for 3 tiles, 72 against 80 for 5, 92 against 101 for 7, 116
// against 124 for 9, 133 against 140 for 11, 155 against 158 for 13, but 84.5
// against 80.4 for 6, 127 against 125 for 10, 191 against 184 for 16.
template <int MODE, bool AH, class Geo>
static cudaError_t round_t(const RoundArgs& ra, const Geo& geo, int64_t N, int per_sm,
                           const uint8_t* packed, unsigned* stw, cudaStream_t st) {
  const int64_t ntiles = (N + TILE - 1) / TILE, sms = num_sms();
  const int64_t each = (ntiles + sms - 1) / sms;
  if (each <= 1) return round_launch<MODE, 4, 1, AH>(ra, geo, (unsigned)ntiles, packed, stw, st);
  if (each == 2 || (each <= 13 && each % 2 == 1))
    return round_launch<MODE, 2, 1, AH>(ra, geo, (unsigned)(ntiles < 2 * sms ? ntiles : 2 * sms),
                                        packed, stw, st);
  // persistent grid: at most per_sm CTAs per SM, each running LBM_ROUND_GROUPS tiles at a time
  const int64_t cta_tiles = (ntiles + LBM_ROUND_GROUPS - 1) / LBM_ROUND_GROUPS;
  const unsigned grid = grid_for(cta_tiles * TILE, per_sm >= 2 ? LBM_ROUND_CTAS : per_sm);
  return round_launch<MODE, LBM_ROUND_TPN, LBM_ROUND_GROUPS, AH>(ra, geo, grid, packed, stw, st);
}

static RoundArgs round_args(const RoundLaunch& rl) {
  return {rl.h_in, rl.ab_in, rl.h_out, rl.a_out, rl.ab_out, rl.y_out, rl.f_post, rl.f_out,
          rl.tau, rl.taus, rl.round, rl.h_skip};
}

// The rounds of an inference step (A recomputed from h): inner round, last
// round + head + Eq. 3.
template <class Geo>
static cudaError_t round_step(int mode, const RoundLaunch& rl, const Geo& geo, int64_t N,
                              const uint8_t* packed, cudaStream_t st, int per_sm = 2) {
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  return mode == 0 ? round_t<0, true>(round_args(rl), geo, N, per_sm, packed, stw, st)
                   : round_t<1, true>(round_args(rl), geo, N, per_sm, packed, stw, st);
}

cudaError_t launch_gnn_encode(const float* f, const Shape& s, const uint8_t* packed,
                              __nv_bfloat16* h0, __half* ab, cudaStream_t st) {
  return encode_t(f, make_geo_stack(s), (int64_t)s.nb * s.ny * s.nx, packed, h0, ab, st);
}

cudaError_t launch_gnn_round(int mode, const RoundLaunch& rl, const Shape& s,
                             const uint8_t* packed, cudaStream_t st) {
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  const GeoStack geo = make_geo_stack(s);
  if (rl.a_from_h) return round_step(mode, rl, geo, N, packed, st);
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  return mode == 0 ? round_t<0, false>(round_args(rl), geo, N, 2, packed, stw, st)
                   : round_t<2, false>(round_args(rl), geo, N, 2, packed, stw, st);
}

// The network forward of the channel (GeoChannel: graph stopped at the
// walls, forced velocity among the features) on pre-collision populations:
// encoder -> h0, A|B of round 0; inner round -> h1, A|B of round 1; last
// round -> the head output y [10][N].  For training, sv.a0, sv.a1 and sv.h2
// (else NULL) receive the aggregated messages and the last node state.
cudaError_t launch_gnn_forward_channel(const float* f_pre, const Shape& s, float force_x,
                                       const float* forces_x, const uint8_t* packed,
                                       const ChannelSaved& sv, float* y, cudaStream_t st) {
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  GeoChannel geo;
  static_cast<GeoStack&>(geo) = make_geo_stack(s);
  geo.fx = force_x;
  geo.fxs = forces_x;
  const int64_t N = (int64_t)s.nb * s.ny * s.nx;
  cudaError_t e;
  if ((e = encode_t(f_pre, geo, N, packed, sv.h0, sv.ab0, st)) != cudaSuccess) return e;
  RoundArgs r0{sv.h0, sv.ab0, sv.h1, sv.a0, sv.ab1, nullptr, nullptr, nullptr, 1.0f, nullptr, 0,
               nullptr};
  if ((e = round_t<0, false>(r0, geo, N, 2, packed, stw, st)) != cudaSuccess) return e;
  RoundArgs r1{sv.h1, sv.ab1, sv.h2, sv.a1, nullptr, y, nullptr, nullptr, 1.0f, nullptr, 1,
               nullptr};
  return round_t<2, false>(r1, geo, N, 2, packed, stw, st);
}

cudaError_t launch_gnn_step_table(const float* f_in, float* f_out, const LatDesc* lat, int first,
                                  int n, const LatBlock* block, int64_t base, int64_t count, int64_t ps,
                                  const uint8_t* packed, __nv_bfloat16* ws, cudaStream_t st,
                                  int per_sm) {
  if (count <= 0) return cudaSuccess;
  const GeoTable geo{lat, first, n, base, count, ps, block};
  __nv_bfloat16* h0 = ws;
  __half* b0 = reinterpret_cast<__half*>(h0 + count * 64);
  __nv_bfloat16* h1 = reinterpret_cast<__nv_bfloat16*>(b0 + count * 64);
  __half* b1 = reinterpret_cast<__half*>(h1 + count * 64);
  cudaError_t e;
  // the whole step of an MLP-only network, or the encoder (gnn_mlp.cu)
  if ((e = launch_gnn_encode_fused_table(f_in, f_out, lat, first, n, block, base, count, ps, packed,
                                         h0, b0, st)) != cudaSuccess)
    return e;
  RoundLaunch r0;
  r0.h_in = h0;
  r0.ab_in = b0;
  r0.a_from_h = true;
  r0.h_skip = h0;
  r0.h_out = h1;
  r0.ab_out = b1;
  r0.round = 0;
  if ((e = round_step(0, r0, geo, count, packed, st, per_sm)) != cudaSuccess) return e;
  RoundLaunch r1;
  r1.h_in = h1;
  r1.ab_in = b1;
  r1.a_from_h = true;
  r1.h_skip = h0;
  r1.f_post = f_in;
  r1.f_out = f_out;
  r1.round = 1;
  return round_step(1, r1, geo, count, packed, st, per_sm);
}

}  // namespace lbmgnn
