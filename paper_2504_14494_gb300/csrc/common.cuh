// Shared device-side definitions of the CUDA library (sm_103a).
//
// D2Q9 lattice (Sec. 2.1 of the paper names w_i and c_s without values; the
// textbook set is used): e_0=(0,0); e_1..4=(1,0),(0,1),(-1,0),(0,-1);
// e_5..8=(1,1),(-1,1),(-1,-1),(1,-1); w = 4/9, 1/9 x4, 1/36 x4; c_s^2 = 1/3.
//
// Population layout: plane q of node (x, y) of lattice b lives at
//   f[q * plane_stride + (b * ny + y) * nx + x]
// i.e. a stack of nb lattices of ny x nx nodes, q-major (SoA), x fastest.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include "../../include/lbmgnn.h"

namespace lbmgnn {

constexpr int Q = 9;
__host__ __device__ constexpr int ex(int i) {
  return (i == 1 || i == 5 || i == 8) ? 1 : (i == 3 || i == 6 || i == 7) ? -1 : 0;
}
__host__ __device__ constexpr int ey(int i) {
  return (i == 2 || i == 5 || i == 6) ? 1 : (i == 4 || i == 7 || i == 8) ? -1 : 0;
}
__host__ __device__ constexpr float wq(int i) {
  return i == 0 ? 4.0f / 9.0f : (i <= 4 ? 1.0f / 9.0f : 1.0f / 36.0f);
}
// the direction opposite to e_i
__host__ __device__ constexpr int opp(int i) {
  return i == 0 ? 0 : (i <= 4 ? ((i + 1) % 4) + 1 : ((i - 5 + 2) % 4) + 5);
}

// Device status word: bit flags raised by kernels, read (and cleared) by
// lbm_get_status().  One per device that loaded the library; kernels receive
// its address as an argument (status_word() returns it for the current
// device).
enum : unsigned {
  ST_NONFINITE = 1u << 0,
  ST_TIMEOUT = 1u << 1,
  ST_BOUNDS = 1u << 2,
  ST_BLOB = 1u << 3,  // a kernel was given a packed parameter image without its validity word
};
unsigned* status_word();

__device__ __forceinline__ void raise_status(unsigned* w, unsigned bits) { atomicOr(w, bits); }

// Bounds-checked builds (-DLBM_BOUNDS_CHECK, liblbmgnn_checked.so): a computed
// gather index outside [lo, hi) raises ST_BOUNDS and is replaced by lo, so
// the access stays inside the buffer and the run goes on; the regular build
// compiles the check away.  (This build, small cases and the oracle stand in
// for a memory checker.)
__device__ __forceinline__ int64_t checked(int64_t i, int64_t lo, int64_t hi, unsigned* stw) {
#ifdef LBM_BOUNDS_CHECK
  if (i < lo || i >= hi) {
    raise_status(stw, ST_BOUNDS);
    return lo;
  }
#endif
  return i;
}

// Moments of one node: rho = sum f_i, (jx, jy) = sum f_i e_i.
struct Moments {
  float rho, ux, uy;
};

__device__ __forceinline__ Moments moments9(const float (&f)[Q]) {
  const float rho = ((f[0] + (f[1] + f[3])) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8]));
  const float jx = (f[1] - f[3]) + (f[5] - f[7]) + (f[8] - f[6]);
  const float jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
  const float inv = 1.0f / rho;
  return {rho, jx * inv, jy * inv};
}

// Eq. 2 for direction i, with c_s^2 = 1/3:
//   f_i^eq = rho w_i (1 + 3 e.u + 9/2 (e.u)^2 - 3/2 u.u)
__device__ __forceinline__ float feq_i(int i, const Moments& m, float usq15) {
  const float eu = float(ex(i)) * m.ux + float(ey(i)) * m.uy;
  return wq(i) * m.rho * (1.0f + 3.0f * eu + 4.5f * eu * eu - usq15);
}

// ---- totals (mass, momentum, kinetic energy) at FP64 accuracy -------------
// GB300 runs FP64 at a small fraction of its FP32 rate, so the per-node sums
// of the totals are carried as unevaluated pairs hi + lo of FP32 values
// ("double-float"): each addition is Knuth's error-free TwoSum (s + e equals
// a + b exactly), the rounding errors collect in lo, and the pair is
// renormalised by another TwoSum once per node.  About 2^-46 relative error
// per node; FP64 arithmetic is used once per warp.
struct DF {
  static constexpr bool kPair = true;
  float hi, lo;
};
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void df_add(DF& a, float x) {  // a += x (lo not renormalised)
  float s, e;
  two_sum(a.hi, x, s, e);
  a.hi = s;
  a.lo = __fadd_rn(a.lo, e);
}
__device__ __forceinline__ void df_norm(DF& a) {
  float s, e;
  two_sum(a.hi, a.lo, s, e);
  a.hi = s;
  a.lo = e;
}
__device__ __forceinline__ void df_add(DF& a, const DF& b) {  // a += b, renormalised
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  a.hi = s;
  a.lo = __fadd_rn(a.lo, __fadd_rn(b.lo, e));
  df_norm(a);
}
__device__ __forceinline__ DF df_shfl_xor(const DF& a, int o) {
  return {__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}

// The sum of a thread that takes many nodes, unevaluated s0 + s1 + s2: s0 and s1
// take error-free sums, s2 collects what s1 rounds off, so that the error does
// not grow with the nodes as that of a DF does (54 equal nodes: up to 2^-46).
// For up to 64 nodes of one sign |s1| <= 2^-17 of the sum, |s2| <= 2^-34 and its
// rounding errors 2^-51.
struct TF {
  static constexpr bool kPair = false;
  float s0 = 0.f, s1 = 0.f, s2 = 0.f;
  __device__ __forceinline__ void add(float hi) {
    float e, g;
    two_sum(s0, hi, s0, e);
    two_sum(s1, e, s1, g);
    s2 = __fadd_rn(s2, g);
  }
  __device__ __forceinline__ void add(const DF& x) {
    float g;
    two_sum(s1, x.lo, s1, g);
    s2 = __fadd_rn(s2, g);
    add(x.hi);
  }
  __device__ __forceinline__ DF pair() const {  // within 2^-48
    DF a;
    two_sum(s0, s1, a.hi, a.lo);
    a.lo = __fadd_rn(a.lo, s2);
    df_norm(a);
    return a;
  }
};

__device__ __forceinline__ void df_add(TF& a, const DF& b) { a.add(b); }
__device__ __forceinline__ DF as_pair(const DF& a) { return a; }
__device__ __forceinline__ DF as_pair(const TF& a) { return a.pair(); }

// Per-thread totals of stored nodes: mass sum f_i, momentum sum f_i e_i,
// kinetic energy sum |j|^2 / (2 rho), and the count of nodes holding a
// non-finite population (excluded from the sums).
// Sum: DF for a few nodes per thread, TF for many.
template <class Sum = DF>
struct NodeTotals {
  Sum sm{}, spx{}, spy{}, se{};
  unsigned bad = 0;

  __device__ __forceinline__ void add(const float (&o)[Q]) {
    bool finite = true;
#pragma unroll
    for (int i = 0; i < Q; ++i) finite &= isfinite(o[i]);
    if (!finite) {
      ++bad;
      return;
    }
    DF r{o[0], 0.f}, jx{0.f, 0.f}, jy{0.f, 0.f};
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      df_add(r, o[i]);
      if (ex(i)) df_add(jx, ex(i) > 0 ? o[i] : -o[i]);
      if (ey(i)) df_add(jy, ey(i) > 0 ? o[i] : -o[i]);
    }
    if constexpr (Sum::kPair) {  // (three words take the node's two as they are)
      df_norm(r);
      df_norm(jx);
      df_norm(jy);
    }
    // (the roundings spelled out: the same in every kernel that takes totals)
    const float rh = __fadd_rn(r.hi, r.lo), jxh = __fadd_rn(jx.hi, jx.lo),
                jyh = __fadd_rn(jy.hi, jy.lo);
    const float en =
        __fdiv_rn(__fmul_rn(0.5f, __fmaf_rn(jxh, jxh, __fmul_rn(jyh, jyh))), rh);
    df_add(sm, r);
    df_add(spx, jx);
    df_add(spy, jy);
    if constexpr (Sum::kPair) df_add(se, DF{en, 0.f}); else se.add(en);
  }

  // Sum over the block (NT threads) added to totals[0..4] in FP64.
  template <int NT>
  __device__ __forceinline__ void flush(double* __restrict__ totals) {
    __shared__ double red[NT / 32][5];
    DF m = as_pair(sm), px = as_pair(spx), py = as_pair(spy), e = as_pair(se);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      df_add(m, df_shfl_xor(m, o));
      df_add(px, df_shfl_xor(px, o));
      df_add(py, df_shfl_xor(py, o));
      df_add(e, df_shfl_xor(e, o));
    }
    const unsigned nbad = __reduce_add_sync(0xffffffffu, bad);
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
      red[w][0] = (double)m.hi + (double)m.lo;
      red[w][1] = (double)px.hi + (double)px.lo;
      red[w][2] = (double)py.hi + (double)py.lo;
      red[w][3] = (double)e.hi + (double)e.lo;
      red[w][4] = (double)nbad;
    }
    __syncthreads();
    if (threadIdx.x < 5) {
      double acc = 0.0;
#pragma unroll
      for (int i = 0; i < NT / 32; ++i) acc += red[i][threadIdx.x];
      if (acc != 0.0) atomicAdd(totals + threadIdx.x, acc);
    }
  }
};

struct Shape {
  int nx, ny, nb;
  int64_t ps;  // plane stride in elements
};

// ---- kernels of one call that overlap at their seams -------------------------
// The kernels of a multi-kernel call are launched with programmatic stream
// serialization (launch_after, launch.h): a kernel starts once every CTA of the
// one before it has passed dep_release(), sets up from what was complete by
// then (the weights), and waits in dep_wait() until the one before it has
// completed and its writes are visible.  Each kernel passes dep_wait() on every
// path, before dep_release(), before it reads anything the one before may have
// written and before it writes anything but the status word, so that "the one
// before has completed" holds for all before it.  gnn_pack, gnn_adamw,
// gnn_backward and gnn_collide_loss launch their first kernel this way too (it
// waits before its first read); the first kernel of every other call is
// launched normally.
// A kernel allocates its tensor memory before dep_release(): CTAs of the next
// kernel allocate theirs before they wait, and one that took columns of an SM
// from a CTA it waits for would block both for good.
__device__ __forceinline__ void dep_wait() {
#if __CUDA_ARCH__ >= 900
  asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
}
__device__ __forceinline__ void dep_release() {
#if __CUDA_ARCH__ >= 900
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
}
__device__ __forceinline__ void dep_sync() {
  dep_wait();
  dep_release();
}

// Reads of what the kernel before may have written.  A kernel launched early
// runs while that one still does, so neither __ldg nor a const __restrict__
// pointer may be used for them: both declare the data unchanged for as long as
// the kernel runs, and such a load may be moved above dep_wait().  ld_prev is a
// plain load; its address depends on an index or a pointer that went through
// after_wait(), which stands after dep_wait(), so that it cannot be moved above
// the wait either.  (Volatile loads keep their order among themselves too: with
// them the message-passing rounds took 3 % longer, the 64 x 256^2 training step
// 1 %.)
template <typename T>
__device__ __forceinline__ T after_wait(T v) {
  static_assert(sizeof(T) == 8 || sizeof(T) == 4, "an index or a pointer");
  if constexpr (sizeof(T) == 8) {
    uint64_t w = (uint64_t)v;
    asm volatile("" : "+l"(w) : : "memory");
    return (T)w;
  } else {
    uint32_t w = (uint32_t)v;
    asm volatile("" : "+r"(w) : : "memory");
    return (T)w;
  }
}
__device__ __forceinline__ float ld_prev(const float* p) {
  float v;
  asm("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double ld_prev(const double* p) {
  double v;
  asm("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ unsigned ld_prev(const unsigned* p) {
  unsigned v;
  asm("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ld_prev(const float4* p) {
  float4 v;
  asm("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ uint4 ld_prev(const uint4* p) {
  uint4 v;
  asm("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
// The read in a kernel that comes in two instances, of which EARLY alone is
// launched early: nothing writes the data while the other one runs.
template <bool EARLY, typename T>
__device__ __forceinline__ T ld_in(const T* p) {
  if constexpr (EARLY)
    return ld_prev(p);
  else
    return __ldg(p);
}

}  // namespace lbmgnn
