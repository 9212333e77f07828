// Several plain steps per launch: the multi-step calls of the BGK step (Eq. 1,
// Eq. 2, Fig. 1 loop) and of the channel step, with the state kept on chip
// between the steps.  Every node of every step is computed by the same BGK
// formula with the same roundings (collide.cuh), or by the same channel_relax, on
// the same nine pulled values as in the single-step kernels, so the results are
// the same bit for bit.
//
// Two forms, chosen by estimated time (launch_bgk_steps):
//
// resident_steps_kernel -- for small lattices and many steps, which are bound
// by the latency of one step: one thread-block cluster (1..16 CTAs) per lattice
// holds the whole lattice in shared memory (two buffers) for all steps of the
// call; per step a pull from shared memory, the collision, a store to the
// other buffer, edge rows also to the neighbouring CTAs' halo rows through
// distributed shared memory.  64^2: 0.41 us a step (4.1 with one launch a
// step); a 4 x 32 channel, in one CTA: 0.23 (4.1).
//
// temporal_steps_kernel -- for larger lattices, which are bound by memory
// traffic (72 bytes per node and step): T = 2..4 steps per pass over memory.
// A strip of 64 columns marches down a range of rows; the rows in flight
// between its T stages stay in registers (and, for small lattices, pass from
// warp to warp through shared memory).  The strip is 4 columns wider on each
// side and the range T rows longer on each side than what is stored (both
// wrap periodically); those are computed redundantly by the neighbours.
// 4096^2: 70 us a step against 175 (72 bytes per node at HBM's rate: 178) --
// bound by FP32 issue (about 100 instructions per node and step) and the 1.2
// times recomputed nodes; 1024^2: 8.4 (10.6); 512^2: 4.2 (6.2); 256^2: 2.6
// (4.2); three odd 1023 x 517: 12.3 (22.8).  Tried on the way: one thread per
// node with all stages handed over in shared memory, 119 at 4096^2; 4 columns
// per lane, 79 to 83 (fewer warps, and the barrier or the registers bind); a
// warp's stages in two independent groups, one a row late, 74 (204 registers).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cooperative_groups.h>
#include <type_traits>

#include "collide.cuh"
#include "launch.h"
#include "umma.cuh"

namespace cg = cooperative_groups;


namespace lbmgnn {

namespace {

__device__ __forceinline__ void cp8(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}

// ---------------------------------------------------------------------------
// Resident form.  CTA r of the cluster holds rows r R .. min(ny, (r + 1) R) - 1
// of lattice b as local rows 1..; local rows 0 and rows + 1 are the halo
// (unused by a CTA that holds the whole lattice).
//
// Between two steps the CTAs of a cluster exchange their edge rows: each edge
// node's three outgoing populations go to the neighbour's halo row by st.async,
// which counts their bytes on an mbarrier there; the threads of the edge rows
// wait for the halo's bytes (an acquire at cluster scope), the others only for
// their own CTA.  (A cluster barrier per step in its place: 0.75 us a step at
// 64^2.)  There is one
// mbarrier per buffer: a CTA cannot start step n + 2 before its neighbours have
// sent step n + 1, so a neighbour is at most one step ahead.
struct ResidentArgs {
  const float* fin;
  float* fout;
  Shape s;
  float tau;
  const float* taus;
  float gx;
  int nsteps;  // >= 1
  int rows;    // R: rows per CTA
};

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_async(uint32_t addr, float v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(
                   addr),
               "r"(__float_as_uint(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void expect_bytes(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

// KN: nodes per thread.  CH: the channel (bounce-back walls, force gx).  ONE:
// the whole lattice in one CTA.
template <bool CH, int KN, bool ONE>
__global__ void __launch_bounds__(1024) resident_steps_kernel(ResidentArgs a, unsigned* stw) {
  extern __shared__ float sm[];
  __shared__ uint64_t bar[2];
  cg::cluster_group cl = cg::this_cluster();
  const int C = ONE ? 1 : (int)cl.num_blocks(), r = ONE ? 0 : (int)cl.block_rank();
  const int nx = a.s.nx, ny = a.s.ny;
  const int64_t b = blockIdx.x / C, lat = b * ny * nx;
  const int ya = r * a.rows, rows = min(ny - ya, a.rows);
  const int pitch = (a.rows + 2) * nx;  // one plane
  const uint32_t halo_bytes = 2u * 3u * 4u * (uint32_t)nx;
  if constexpr (!ONE) {
    if (threadIdx.x == 0) {
      mbar_init(&bar[0], 1);
      mbar_init(&bar[1], 1);
      expect_bytes(&bar[0], halo_bytes);
      expect_bytes(&bar[1], halo_bytes);
    }
  }
  // the neighbours (periodic): the CTA holding row ya - 1 and the one holding
  // row ya + rows, and the local index of the halo row this CTA fills there
  const int up = r == 0 ? C - 1 : r - 1, dn = r == C - 1 ? 0 : r + 1;
  const int up_rows = min(ny - up * a.rows, a.rows);
  const uint32_t up_sm = map_rank(smem_u32(sm), up), dn_sm = map_rank(smem_u32(sm), dn);
  const uint32_t up_bar = map_rank(smem_u32(bar), up), dn_bar = map_rank(smem_u32(bar), dn);
  const float* fin = a.fin + lat;
  // own rows and both halo rows
  for (int i = threadIdx.x; i < (rows + 2) * nx; i += blockDim.x) {
    const int ly = i / nx, x = i - ly * nx;
    int y = ya + ly - 1;
    y = y < 0 ? ny - 1 : (y >= ny ? 0 : y);
#pragma unroll
    for (int q = 0; q < Q; ++q)
      sm[q * pitch + i] = __ldg(
          fin + q * a.s.ps + checked((int64_t)y * nx + x, 0, (int64_t)ny * nx, stw));
  }
  // this thread's nodes: own offset, and the sources of the nine populations
  int own[KN], src[KN][Q];
  bool first_row[KN], last_row[KN];
#pragma unroll
  for (int k = 0; k < KN; ++k) {
    const int i = threadIdx.x + k * blockDim.x;
    const int ly = i < rows * nx ? i / nx : -1;
    const int x = ly < 0 ? 0 : i - ly * nx, y = ya + ly;
    first_row[k] = ly == 0;
    last_row[k] = ly == rows - 1;
    own[k] = ly < 0 ? -1 : (ly + 1) * nx + x;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      int xs = x - ex(q), ls = ly + 1 - ey(q);
      xs = xs < 0 ? nx - 1 : (xs >= nx ? 0 : xs);
      if (ONE && !CH) ls = ls < 1 ? rows : (ls > rows ? 1 : ls);
      src[k][q] = q * pitch + ls * nx + xs;
      if (CH && (y - ey(q) < 0 || y - ey(q) >= ny)) src[k][q] = opp(q) * pitch + own[k];  // bounce-back
      if (ly < 0) src[k][q] = 0;
    }
  }
  const float tau = a.taus ? __ldg(a.taus + b) : a.tau;
  const float omega = 1.0f / tau;
  if constexpr (ONE) __syncthreads(); else cl.sync();

  int cur = 0, nxt = Q * pitch;
  for (int step = 0; step < a.nsteps; ++step) {
    const bool last = step == a.nsteps - 1;
    bool lost = false;  // a neighbour's rows never came
#pragma unroll
    for (int k = 0; k < KN; ++k) {
      if (own[k] < 0) continue;
      if constexpr (!ONE) {
        // the halo of this step's buffer (step 0: loaded above)
        if (step > 0 && (first_row[k] || last_row[k])) {
          const int h = step & 1;  // filled during step - 1
          if (!mbar_wait<true>(&bar[h], ((step - 1) >> 1) & 1)) lost = true;
          if (k == 0 && threadIdx.x == 0) expect_bytes(&bar[h], halo_bytes);  // for step + 2
        }
      }
      float f[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) f[q] = sm[cur + src[k][q]];
      if constexpr (CH) channel_relax<true>(f, tau, a.gx); else bgk_collide_fast(f, omega);
      if (last) {
        float* o = a.fout + lat + (int64_t)(ya - 1) * nx + own[k];
#pragma unroll
        for (int q = 0; q < Q; ++q) o[q * a.s.ps] = f[q];
      } else {
        float* o = sm + nxt + own[k];
#pragma unroll
        for (int q = 0; q < Q; ++q) o[q * pitch] = f[q];
        if constexpr (!ONE) {
          // the rows the neighbours pull across the cut (across the channel's
          // walls too, where nothing reads them: the byte counts stay alike)
          const uint32_t h = 8u * ((step + 1) & 1);
          if (first_row[k]) {  // e_y = -1: below the last row of `up`
            const uint32_t o4 = up_sm + 4u * (nxt + own[k] + up_rows * nx);
            st_async(o4 + 16u * pitch, f[4], up_bar + h);
            st_async(o4 + 28u * pitch, f[7], up_bar + h);
            st_async(o4 + 32u * pitch, f[8], up_bar + h);
          }
          if (last_row[k]) {  // e_y = +1: above the first row of `dn`
            const uint32_t o4 = dn_sm + 4u * (nxt + own[k] - rows * nx);
            st_async(o4 + 8u * pitch, f[2], dn_bar + h);
            st_async(o4 + 20u * pitch, f[5], dn_bar + h);
            st_async(o4 + 24u * pitch, f[6], dn_bar + h);
          }
        }
      }
    }
    if constexpr (ONE) {
      __syncthreads();
    } else if (__syncthreads_or(lost)) {
      if (threadIdx.x == 0) raise_status(stw, ST_TIMEOUT);
      break;
    }
    const int t = cur;
    cur = nxt;
    nxt = t;
  }
  // no CTA leaves while a neighbour may still reach into its shared memory
  if constexpr (!ONE) cl.sync();
}

constexpr int SMEM_MAX = 227 * 1024 - 64;  // (64: the mbarriers)

uint32_t resident_smem(int rows, int nx) { return 2u * Q * (uint32_t)(rows + 2) * nx * 4u; }

// Cluster size (the largest up to C that leaves no CTA without rows) and rows
// per CTA, or C = 0 when the lattice does not fit.
struct ResidentPlan {
  int C, rows, threads, kn;
};
ResidentPlan plan_resident_from(const Shape& s, int C) {
  for (; C >= 1; C >>= 1) {
    if (C > s.ny) continue;
    const int rows = (s.ny + C - 1) / C;
    if ((int64_t)rows * (C - 1) >= s.ny) continue;  // a CTA without rows
    const int nodes = rows * s.nx;
    const int kn = (nodes + 1023) / 1024;
    if (kn > 3 || resident_smem(rows, s.nx) > (uint32_t)SMEM_MAX) break;
    return {C, rows, ((nodes + kn - 1) / kn + 31) / 32 * 32, kn};
  }
  return {0, 0, 0, 0};
}

template <bool CH, int KN, bool ONE>
cudaError_t resident_t(const ResidentArgs& a, const ResidentPlan& p, cudaStream_t st) {
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  const uint32_t bytes = resident_smem(p.rows, a.s.nx);
  auto* kern = resident_steps_kernel<CH, KN, ONE>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  if (p.C > 8 && (e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                           1)) != cudaSuccess)
    return e;
  cfg.gridDim = dim3((unsigned)p.C * (unsigned)a.s.nb);
  cfg.blockDim = dim3((unsigned)p.threads);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)p.C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a, stw);
}

template <bool CH>
cudaError_t resident(const ResidentArgs& a, const ResidentPlan& p, cudaStream_t st) {
  if (p.C == 1) {
    switch (p.kn) {
      case 1: return resident_t<CH, 1, true>(a, p, st);
      case 2: return resident_t<CH, 2, true>(a, p, st);
      // (one CTA takes at most 512 nodes, or one row, of which 1,075 nodes fit)
      default: return cudaErrorInvalidConfiguration;
    }
  }
  switch (p.kn) {
    case 1: return resident_t<CH, 1, false>(a, p, st);
    case 2: return resident_t<CH, 2, false>(a, p, st);
    default: return resident_t<CH, 3, false>(a, p, st);
  }
}

// ---------------------------------------------------------------------------
// Temporal form.  A CTA owns a strip of 64 columns (2 per lane, one packed
// pair) and a range of rows.  Its T steps are T stages, S of them in each of
// G = T / S warps: a stage receives the rows of the step before it one after
// the other, keeps the two rows it still needs in registers, and passes its
// own row on, in registers to the next stage of its warp or through shared
// memory to the next warp.
constexpr int COLS = 64;
constexpr int HALO = 4;              // columns computed redundantly on each side (>= T)
constexpr int AHEAD = 2;             // input rows in flight
constexpr int RING = AHEAD + 1;      // input row ring
constexpr int ROWF = Q * COLS;       // floats of one row

struct TemporalArgs {
  const float* fin;
  float* fout;
  Shape s;
  float tau;
  const float* taus;
  int strips;                // strips of COLS - 2 HALO columns (the last may be narrower)
  int segs, height;          // row ranges of `height` rows
  int64_t units;             // nb * strips * segs
};

// Strips per CTA (four independent warps when one warp holds all stages) and
// resident CTAs per SM: 12 warps of 168 registers (all stages in one warp) or
// 24 warps of 80 (one stage per warp).
template <int G>
constexpr int temporal_units() {
  return G == 1 ? 4 : 1;
}
template <int G>
constexpr int temporal_ctas() {
  return G == 1 ? 3 : 24 / G;
}

// Shared memory in rows of ROWF floats: the input ring, then two slots per
// hand-over between warps, then (!VEC) the row being stored.
template <int G, bool VEC>
constexpr int temporal_bytes() {
  return temporal_units<G>() * (RING + 2 * (G - 1) + (VEC ? 0 : 1)) * ROWF * 4;
}
// VEC: nx % 2 == 0 and 8-byte aligned planes (8-byte copies and stores;
// 16-byte copies, half a warp per plane, took 7 to 45 % longer); otherwise
// columns move one by one, stores through shared memory.
template <int T, int S, bool VEC>
__global__ void __launch_bounds__(32 * (T / S) * temporal_units<T / S>(),
                                  temporal_ctas<T / S>()) temporal_steps_kernel(
    TemporalArgs a, unsigned* stw) {
  constexpr int G = T / S;
  constexpr int U = temporal_units<G>();
  extern __shared__ float4 sm4[];
  const int lane = threadIdx.x & 31, w = G == 1 ? 0 : threadIdx.x >> 5;
  const int sub = G == 1 ? threadIdx.x >> 5 : 0;
  float* sm = reinterpret_cast<float*>(sm4) + sub * (temporal_bytes<G, VEC>() / (4 * U));
  const int64_t unit = (int64_t)blockIdx.x * U + sub;
  if (unit >= a.units) return;  // (U > 1 only: no block-wide barrier below)
  const int nx = a.s.nx, ny = a.s.ny;
  const int seg = (int)(unit % a.segs);
  const int64_t bs = unit / a.segs;
  const int strip = (int)(bs % a.strips);
  const int64_t b = bs / a.strips;
  const int x0 = strip * (COLS - 2 * HALO), y0 = seg * a.height;
  const int height = min(a.height, ny - y0);
  const int K = height + 2 * T;  // input rows 0..K-1: lattice row y0 - T + k (periodic)
  auto wrap = [](int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
  };
  // source columns: 2 consecutive ones (VEC) or lane + 32 j
  int xs[VEC ? 1 : 2];
#pragma unroll
  for (int j = 0; j < (VEC ? 1 : 2); ++j)
    xs[j] = wrap(x0 - HALO + (VEC ? 2 * lane : lane + 32 * j), nx);
  int yin = wrap(y0 - T, ny);
  const float* fin = a.fin + b * ny * nx;
  const int64_t lat_nodes = (int64_t)ny * nx, ps = a.s.ps;
  const float om = -(1.0f / (a.taus ? __ldg(a.taus + b) : a.tau));
  const float2 nomega = make_float2(om, om);

  auto fetch = [&](int k) {  // warp 0: input row k -> ring
    if (k < K) {
      float* d = sm + (k % RING) * ROWF;
      if constexpr (VEC) {
        const int64_t o = checked((int64_t)yin * nx + xs[0], 0, lat_nodes - 1, stw);
#pragma unroll
        for (int q = 0; q < Q; ++q) cp8(d + q * COLS + 2 * lane, fin + q * ps + o);
      } else {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int64_t o = checked((int64_t)yin * nx + xs[j], 0, lat_nodes, stw);
#pragma unroll
          for (int q = 0; q < Q; ++q) cp4(d + q * COLS + lane + 32 * j, fin + q * ps + o);
        }
      }
      yin = yin + 1 == ny ? 0 : yin + 1;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (w == 0) {
    for (int k = 0; k < AHEAD; ++k) fetch(k);
  }
  // hand-over slots into and out of this warp; the row being stored (!VEC)
  const float* in_slot = sm + (RING + 2 * (w - 1)) * ROWF + 2 * lane;
  float* out_slot = sm + (RING + 2 * w) * ROWF + 2 * lane;
  float* stage_out = sm + (RING + 2 * (G - 1)) * ROWF;
  // where the last stage stores: 2 consecutive columns, or lane + 32 j
  float* out = a.fout + b * ny * nx + (int64_t)y0 * nx + x0 - HALO;
  const bool vstore = 2 * lane >= HALO && 2 * lane < COLS - HALO && x0 - HALO + 2 * lane < nx;

  // Per stage, z: the e_y = 0 populations of the row received last; p: the
  // e_y = +1 populations of the last two rows (all already shifted by e_x).
  float2 z[S][3], p[S][2][3];
#pragma unroll
  for (int s = 0; s < S; ++s)
#pragma unroll
    for (int j = 0; j < 3; ++j) z[s][j] = p[s][0][j] = p[s][1][j] = make_float2(0.1f, 0.1f);

  // Iteration i: warp w receives row i - (S + 1) w of its input (row k of
  // any step is the input row k's lattice row) and each of its stages
  // computes the row before the one it receives.  PAR = i & 1 selects the
  // hand-over slots and the p row to replace.
  auto iteration = [&](int i, auto par) {
    constexpr int PAR = decltype(par)::value;
    float2 f[Q];
    if (w == 0) {
      asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD - 1) : "memory");
      __syncwarp();  // every lane's copies of row i have landed
    }
    {
      const float* r = w == 0 ? sm + (i % RING) * ROWF + 2 * lane : in_slot + (1 - PAR) * ROWF;
#pragma unroll
      for (int q = 0; q < Q; ++q) f[q] = *reinterpret_cast<const float2*>(r + q * COLS);
    }
    if (w == 0) fetch(i + AHEAD);  // into the slot of row i - 1, which every lane has read
#pragma unroll
    for (int s = 0; s < S; ++s) {
      // shift by e_x (the strip's outer columns take whatever the edge lanes
      // hold: they are never stored)
      float2 g[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        g[q] = f[q];
        if (ex(q) > 0)
          g[q] = make_float2(__shfl_up_sync(0xffffffffu, g[q].y, 1), g[q].x);
        else if (ex(q) < 0)
          g[q] = make_float2(g[q].y, __shfl_down_sync(0xffffffffu, g[q].x, 1));
      }
      // e_y = -1 from the row just received, e_y = 0 from the one before it,
      // e_y = +1 from the one before that
      f[0] = z[s][0], f[1] = z[s][1], f[3] = z[s][2];
      f[2] = p[s][PAR][0], f[5] = p[s][PAR][1], f[6] = p[s][PAR][2];
      f[4] = g[4], f[7] = g[7], f[8] = g[8];
      z[s][0] = g[0], z[s][1] = g[1], z[s][2] = g[3];
      p[s][PAR][0] = g[2], p[s][PAR][1] = g[5], p[s][PAR][2] = g[6];
      bgk_collide_pair(f, nomega);
    }
    if (w < G - 1) {
      float* o = out_slot + PAR * ROWF;
#pragma unroll
      for (int q = 0; q < Q; ++q) *reinterpret_cast<float2*>(o + q * COLS) = f[q];
    } else if (i >= 2 * T + G - 1) {  // lattice row y0 + i - (2 T + G - 1)
      float* o = out + (int64_t)(i - (2 * T + G - 1)) * nx;
      if constexpr (VEC) {
        if (vstore) {
#pragma unroll
          for (int q = 0; q < Q; ++q) *reinterpret_cast<float2*>(o + q * ps + 2 * lane) = f[q];
        }
      } else {
        __syncwarp();
#pragma unroll
        for (int q = 0; q < Q; ++q)
          *reinterpret_cast<float2*>(stage_out + q * COLS + 2 * lane) = f[q];
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int cc = lane + 32 * j;
          if (cc >= HALO && cc < COLS - HALO && x0 - HALO + cc < nx) {
#pragma unroll
            for (int q = 0; q < Q; ++q) o[q * ps + cc] = stage_out[q * COLS + cc];
          }
        }
      }
    }
    if constexpr (G > 1) __syncthreads();
  };
  const int iters = K + G - 1;
  for (int i = 0; i < iters; i += 2) {
    iteration(i, std::integral_constant<int, 0>{});
    if (i + 1 < iters) iteration(i + 1, std::integral_constant<int, 1>{});
  }
}

template <int T, int S, bool VEC>
cudaError_t temporal_t(TemporalArgs a, cudaStream_t st) {
  constexpr int G = T / S, U = temporal_units<G>();
  unsigned* stw = status_word();
  if (!stw) return cudaErrorInvalidDevice;
  temporal_steps_kernel<T, S, VEC>
      <<<(unsigned)((a.units + U - 1) / U), 32 * G * U, temporal_bytes<G, VEC>(), st>>>(a, stw);
  return cudaGetLastError();
}

// ---- which form -------------------------------------------------------------
// Estimated times in microseconds, fitted to sweeps of 32^2 .. 4096^2 lattices
// and stacks on a GB300 (152 SMs): a step of the single-step kernel (4.1 per
// launch; 7.3e-6 per node out of L2, 10.45e-6 out of HBM), a step of the
// resident form, and a pass of the temporal form.  They only rank the forms.
//
// Captured launches (`cap`) cost less than those the host makes one by one, a
// single step of a small lattice 2.3 instead of 4.1, so that more calls are
// best made of single steps: a 200^2 channel's 5 steps 14 us in a graph, 23 by
// the resident form (eager: 21 and 25); 512^2 BGK, 10 steps, 38 and 39 (62 and
// 45).
bool is_captured(cudaStream_t st) {
  cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &c) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return c != cudaStreamCaptureStatusNone;
}

double single_us(const Shape& s, bool cap) {
  const double n = (double)s.nb * s.ny * s.nx;
  return cap ? std::max({2.3, 1.9 + 7.0e-6 * n, 10.45e-6 * n})
             : std::max({4.1, 3.0 + 7.3e-6 * n, 10.45e-6 * n});
}

// Clusters of 16 CTAs (more than every device takes) that run at once on this
// one, at the kernel's most threads and shared memory; 0: none.
int clusters16() {
  static std::atomic<int> cached[64];  // + 1
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int n = cached[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    auto* kern = resident_steps_kernel<false, 1, false>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(1024);
    cfg.dynamicSmemBytes = SMEM_MAX;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 16;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int most = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX) !=
            cudaSuccess ||
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&most, kern, &cfg) != cudaSuccess) {
      cudaGetLastError();
      most = 0;
    }
    n = most + 1;
    cached[dev].store(n, std::memory_order_relaxed);
  }
  return n - 1;
}

// `nsteps` steps of the resident form: 4 for the launch; per wave of clusters
// (about 16 of 8 CTAs run at once, of 16 CTAs what the device says) 4 to load
// and store; per step the chain of one node and the exchange, and the nodes of
// a CTA (more than one per thread at half the rate; clusters of 16 fitted by
// themselves: 64^2, 100 x 96, 128^2, 200^2).  The channel's collision (`ch`)
// takes 1.3 to 1.5 times as long per node: a step of 200^2 3.25 us against 2.6,
// of 128^2 1.14 against 0.86, of 100^2 1.87 against 1.38; its stacks are counted
// with the CTAs that share an SM (64 registers per thread).
double resident_us(const Shape& s, const ResidentPlan& p, int nsteps, bool ch, bool cap) {
  int at_once = p.C == 16 ? std::max(1, clusters16()) : 128 / p.C;
  if (ch && p.C < 16)
    at_once *= std::max(1, std::min(1024 / p.threads, (int)(SMEM_MAX / resident_smem(p.rows, s.nx))));
  const double waves = (double)((s.nb + at_once - 1) / at_once);
  const double nodes = (double)p.rows * s.nx;
  const double one = ch ? (p.C == 16 ? 0.88e-3 : 0.42e-3) : (p.C == 16 ? 0.64e-3 : 0.31e-3);
  const double more = ch ? (p.C == 16 ? 1.16e-3 : 1.13e-3) : (p.C == 16 ? 0.91e-3 : 0.73e-3);
  const double node = (p.kn == 1 ? one : more) * nodes;
  const double step =
      p.C == 16 ? std::max(0.37, 0.24 + node) : (p.C == 1 ? 0.20 : 0.38) + node;
  return (cap ? 0.0 : 4.0) + waves * ((cap ? 3.3 : 4.0) + nsteps * step);
}

// The fastest by that estimate.  One CTA up to 512 nodes without an exchange
// beats several (8 x 32 channel: 0.26 us a step against 0.44).  Clusters of 16
// halve the nodes of a CTA: 64^2 0.41 us a step against 0.53 in clusters of 8,
// 128^2 1.09 against 2.08 (several steps per pass), four 100 x 96 1.05 against
// 1.69; at 32^2 nothing is left to halve (0.38 against 0.36), and fewer run at
// once (one per GPC), so that stacks stay with 8.
ResidentPlan plan_resident(const Shape& s, int nsteps, bool ch, bool cap) {
  const int64_t all = (int64_t)s.nx * s.ny;
  if (all > 16 * 3072) return {0, 0, 0, 0};
  ResidentPlan p = plan_resident_from(s, all <= 512 ? 1 : 8);
  if (all > 1024 && s.ny >= 16 && clusters16() > 0) {
    const ResidentPlan w = plan_resident_from(s, 16);
    if (w.C == 16 &&
        (!p.C || resident_us(s, w, nsteps, ch, cap) < resident_us(s, p, nsteps, ch, cap)))
      p = w;
  }
  return p;
}

struct TemporalPlan {
  double us = 1e30;  // per pass
  bool one = false;  // all stages in one warp
  int strips = 0, segs = 0, height = 0;
};

// A pass of T steps: 4.5 for the launch and the first row, and per row an
// iteration whose time depends on the warps that share the SM (one stage per
// warp: 0.33 alone, 0.89 at 24 warps; four stages in one warp: 0.65 alone,
// 1.54 at 12), at least what HBM takes for the state once in and out.  The
// range heights tried are those that give 1, 2, .. CTAs per SM and whole
// waves: short ranges fill the SMs, long ones recompute fewer rows.  Captured: 2
// less for the launch, but up to 2.5 more between 50 and 500 thousand nodes,
// where an eager pass hides them behind its launch.
TemporalPlan plan_temporal(const Shape& s, int T, int sms, bool cap) {
  TemporalPlan best;
  const int strips = (s.nx + COLS - 2 * HALO - 1) / (COLS - 2 * HALO);
  const int64_t cols = (int64_t)s.nb * strips;
  const double nodes = (double)s.nb * s.ny * s.nx;
  const double fixed =
      cap ? 2.5 + std::min(2.5, 6e-6 * std::max(0.0, nodes - 5e4)) : 4.5;
  for (int form = 0; form < 2; ++form) {
    const bool one = form == 0;
    const int most = one ? 12 : 24 / T;           // strips' CTAs (warps) per SM
    // warps (one) or CTAs per SM aimed at, then two and three whole waves
    const int step = one ? 4 : 1, tries = most / step + 2;
    for (int k = 1; k <= tries; ++k) {
      const int want = k * step <= most ? k * step : (k - most / step + 1) * most;
      const int64_t segs_want = std::max<int64_t>(1, (int64_t)sms * want / cols);
      const int h = (int)((s.ny + std::min<int64_t>(segs_want, s.ny) - 1) /
                          std::min<int64_t>(segs_want, s.ny));
      const int segs = (s.ny + h - 1) / h;
      const int64_t n = cols * segs;
      const double per_sm = (double)((n + sms - 1) / sms);
      const double waves = std::max(1.0, std::ceil(per_sm / most));
      const double warps = std::min(per_sm, (double)most) * (one ? 1 : T);
      const double it = one ? std::max(0.25 + 0.1 * T, 0.25 * T * (0.25 + 0.108 * warps))
                            : std::max(0.33, 0.22 + 0.0278 * warps);
      const double us =
          std::max(fixed + waves * it * (h + 2 * T + (one ? 0 : T - 1)), 13.5e-6 * nodes);  // (HBM)
      if (us < best.us) best = {us, one, strips, segs, h};
    }
  }
  return best;
}

template <int T>
cudaError_t temporal(const float* src, float* dst, const Shape& s, float tau, const float* taus,
                     const TemporalPlan& p, cudaStream_t st) {
  const TemporalArgs a{src, dst, s, tau, taus, p.strips, p.segs, p.height,
                       (int64_t)s.nb * p.strips * p.segs};
  const bool vec = s.nx % 2 == 0 && s.ps % 2 == 0 && ((uintptr_t)src | (uintptr_t)dst) % 8 == 0;
  if (p.one) return vec ? temporal_t<T, T, true>(a, st) : temporal_t<T, T, false>(a, st);
  return vec ? temporal_t<T, 1, true>(a, st) : temporal_t<T, 1, false>(a, st);
}

// `nsteps` steps as one resident launch or as passes of 1 to MOST steps: the
// fewest microseconds in all, for the last ones (up to TAIL) exactly, before
// them passes of the cheapest kind per step.
constexpr int MOST = 4, TAIL = 12;
struct StepsPlan {
  double us = 0.0;
  ResidentPlan resident{0, 0, 0, 0};  // C = 0: by passes
  TemporalPlan pass[MOST + 1];
  int head = 0, head_steps = 1, tail = 0, passes = 0;  // head passes of head_steps, then `tail` steps
  int first[TAIL + 1] = {0};                            // steps of the next pass with n left
};
StepsPlan plan_steps(const Shape& s, int nsteps, int sms, bool cap) {
  StepsPlan p;
  double us[MOST + 1] = {0.0, single_us(s, cap)};
  const bool wide = s.nx >= (1 << 30) || s.ny >= (1 << 30);  // 32-bit rows and columns
  for (int T = 2; T <= MOST && T <= nsteps; ++T) {
    if (!wide) p.pass[T] = plan_temporal(s, T, sms, cap);
    us[T] = p.pass[T].us;
    if (us[T] / T < us[p.head_steps] / p.head_steps) p.head_steps = T;
  }
  p.tail = nsteps;
  if (nsteps > TAIL) {
    p.head = (nsteps - TAIL + p.head_steps - 1) / p.head_steps;
    p.tail -= p.head * p.head_steps;
  }
  double cost[TAIL + 1] = {0.0};
  for (int n = 1; n <= p.tail; ++n) {
    cost[n] = 1e30;
    for (int T = 1; T <= MOST && T <= n; ++T)
      if (cost[n - T] + us[T] < cost[n]) cost[n] = cost[n - T] + us[T], p.first[n] = T;
  }
  p.us = p.head * us[p.head_steps] + cost[p.tail];
  p.passes = p.head;
  for (int n = p.tail; n > 0; n -= p.first[n]) ++p.passes;
  if (nsteps > 1) {
    const ResidentPlan rp = plan_resident(s, nsteps, false, cap);
    const double rus = rp.C ? resident_us(s, rp, nsteps, false, cap) : 1e30;
    if (rus < p.us) p.us = rus, p.resident = rp;
  }
  return p;
}

cudaError_t run_steps(const StepsPlan& p, const float* fin, float* fout, float* ftmp,
                      const Shape& s, float tau, const float* taus, int nsteps, cudaStream_t st) {
  if (p.resident.C) {
    const ResidentArgs a{fin, fout, s, tau, taus, 0.0f, nsteps, p.resident.rows};
    return resident<false>(a, p.resident, st);
  }
  // ping-pong so that the last pass lands in fout
  const float* src = fin;
  int left = p.tail;
  for (int k = 0; k < p.passes; ++k) {
    const int T = k < p.head ? p.head_steps : p.first[left];
    if (k >= p.head) left -= T;
    float* dst = (p.passes - k) % 2 == 1 ? fout : ftmp;
    cudaError_t e = cudaSuccess;
    switch (T) {
      case 1: e = launch_bgk_step(src, dst, s, tau, taus, nullptr, st); break;
      case 2: e = temporal<2>(src, dst, s, tau, taus, p.pass[2], st); break;
      case 3: e = temporal<3>(src, dst, s, tau, taus, p.pass[3], st); break;
      default: e = temporal<4>(src, dst, s, tau, taus, p.pass[4], st); break;
    }
    if (e != cudaSuccess) return e;
    src = dst;
  }
  return cudaSuccess;
}

// What totals add: a pass of the moments kernel over the final state, or, to a
// single step that takes them along, 5 atomics per block.
double moments_us(double n) { return std::min(4.0 + 28e-6 * n, 9.0 + 10e-6 * n); }
double fused_totals_us(double blocks) { return 2.8 + 5e-3 * blocks; }

}  // namespace

int sm_count() {
  static std::atomic<int> cached[64];
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  n = cached[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    cached[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

// With totals the last step may be a single one that takes them along: better
// for few steps of a small lattice (512^2, 2 steps: 17 us against 24 with a
// pass for the totals after both), while a pass pays where it costs less than
// the atomics of a single step and what that step would save inside a pass of
// several (2048^2, 4096^2, 1.6 M odd nodes).
cudaError_t launch_bgk_steps(const float* fin, float* fout, float* ftmp, const Shape& s, float tau,
                             const float* taus, int nsteps, double* totals, cudaStream_t st) {
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidDevice;
  const bool cap = is_captured(st);
  const StepsPlan all = plan_steps(s, nsteps, sms, cap);
  if (totals) {
    const double n = (double)s.nb * s.ny * s.nx;
    const StepsPlan but_one = plan_steps(s, nsteps - 1, sms, cap);
    const double blocks = (double)bgk_step_blocks(ftmp, fout, s);
    if (but_one.us + single_us(s, cap) + fused_totals_us(blocks) < all.us + moments_us(n)) {
      const cudaError_t e = run_steps(but_one, fin, ftmp, fout, s, tau, taus, nsteps - 1, st);
      return e != cudaSuccess ? e : launch_bgk_step(ftmp, fout, s, tau, taus, totals, st);
    }
  }
  const cudaError_t e = run_steps(all, fin, fout, ftmp, s, tau, taus, nsteps, st);
  return e != cudaSuccess || !totals
             ? e
             : launch_moments(fout, s, nullptr, nullptr, nullptr, totals, st);
}

// The channel has the resident form alone; its single-step kernel takes 4.2 a
// launch (and 4 for the first; captured 2.5), 16.7e-6 per node.
bool channel_steps_fit(const Shape& s, int nsteps, cudaStream_t st) {
  const bool cap = is_captured(st);
  const ResidentPlan rp = plan_resident(s, nsteps, true, cap);
  const double n = (double)s.nb * s.ny * s.nx;
  const double singles = cap ? nsteps * std::max({2.5, 2.2 + 15.5e-6 * n, 16.7e-6 * n})
                             : 4.0 + nsteps * std::max(4.2, 16.7e-6 * n);
  return rp.C != 0 && 1.1 * resident_us(s, rp, nsteps, true, cap) < singles;
}

cudaError_t launch_channel_steps(const float* fin, float* fout, const Shape& s, float tau,
                                 const float* taus, float gx, int nsteps, cudaStream_t st) {
  const ResidentPlan rp = plan_resident(s, nsteps, true, is_captured(st));
  if (!rp.C) return cudaErrorInvalidValue;
  const ResidentArgs a{fin, fout, s, tau, taus, gx, nsteps, rp.rows};
  return resident<true>(a, rp, st);
}

}  // namespace lbmgnn
