// Self-tests: the bounded device waits (failure detection), and the reciprocals
// of the collisions.
//
// Failure-detection self-test of the bounded device waits.  Every wait of
// the tensor-core kernels on an mbarrier gives up after a cycle budget,
// raises the timeout bit of the status word and lets the kernel release its
// resources and return.  This kernel exercises exactly that path on a barrier
// that nothing ever arrives on, with a short budget; nothing traps or hangs.
#include "collide.cuh"
#include "umma.cuh"

namespace lbmgnn {

__global__ void wait_timeout_kernel(long long max_cycles, unsigned* stw, int* gave_up) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) mbar_init(&bar, 1);
  __syncthreads();
  const bool ok = mbar_wait(&bar, 0, max_cycles);  // no arrival: must give up
  if (__syncthreads_or(!ok) && threadIdx.x == 0) {
    raise_status(stw, ST_TIMEOUT);
    if (gave_up) *gave_up = 1;
  }
}

// Every float against the IEEE quotient: bad[0] counts the values of rcp2_mid's
// range (|x| in [2^-100, 2^100], both signs) it is not equal for, bad[1] the
// floats (all 2^32) for which rcp1 is neither equal nor NaN with the quotient.
__global__ void __launch_bounds__(256) reciprocal_kernel(unsigned long long* bad) {
  unsigned long long mid = 0, any = 0;
  const uint64_t nth = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (uint64_t(1) << 32);
       i += nth) {
    const float x = __uint_as_float((uint32_t)i), want = 1.0f / x;
    const unsigned w = __float_as_uint(want), got = __float_as_uint(rcp1(x));
    any += got != w && !(isnan(want) && isnan(__uint_as_float(got)));
    if (fabsf(x) >= 0x1p-100f && fabsf(x) <= 0x1p100f) {
      const float2 r = rcp2_mid(make_float2(x, -x));
      mid += __float_as_uint(r.x) != w || __float_as_uint(r.y) != (w ^ 0x80000000u);
    }
  }
  if (mid) atomicAdd(bad, mid);
  if (any) atomicAdd(bad + 1, any);
}

}  // namespace lbmgnn

extern "C" int lbm_selftest_reciprocal(unsigned long long* bad, void* stream) {
  using namespace lbmgnn;
  if (!bad) return LBM_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(bad, 0, 2 * sizeof(*bad), st) != cudaSuccess) return LBM_ERR_CUDA;
  reciprocal_kernel<<<4096, 256, 0, st>>>(bad);
  return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

extern "C" int lbm_selftest_wait_timeout(long long max_cycles, void* stream) {
  using namespace lbmgnn;
  if (max_cycles < 1 || max_cycles > 2000000000LL) return LBM_ERR_ARG;
  unsigned* stw = status_word();
  if (!stw) return LBM_ERR_CUDA;
  wait_timeout_kernel<<<1, 64, 0, static_cast<cudaStream_t>(stream)>>>(max_cycles, stw, nullptr);
  return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}
