// The single-precision operations of the catalog recipe (csrc/generate.cuh) against the IEEE ones,
// compiled and called by test_gpu_gen_arith.py.  Each function returns the count of differences
// over its range, or -1 after a CUDA error.
#include <cuda_runtime.h>

#include "generate.cuh"

using namespace gbsub;

namespace {

constexpr unsigned kMant = 1u << 23;

__device__ float make(unsigned mantissa, int e, unsigned sign = 0) {
  return __uint_as_float(sign << 31 | (unsigned)(e + 127) << 23 | mantissa);
}
__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b); }

// what: 0 reciprocal, 1 square root, 2 x / ln 2, 3 quotients of every divisor mantissa
template <int what>
__global__ void k_count(int e0, int e1, unsigned long long* bad) {
  const unsigned m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= kMant) return;
  unsigned n = 0;
  for (int e = e0; e <= e1; ++e) {
    const float x = make(m, e);
    if (what == 0) n += !same(gen_rcp(x), __frcp_rn(x)) + !same(gen_rcp(-x), __frcp_rn(-x));
    if (what == 1) n += !same(gen_sqrt(x), __fsqrt_rn(x));
    if (what == 2) {
      const float ln2 = (float)0.6931471805599453;
      n += !same(gen_div_ln2(x), __fdiv_rn(x, ln2)) + !same(gen_div_ln2(-x), __fdiv_rn(-x, ln2));
    }
    if (what == 3) {
      // dividends from a counter-based generator
      unsigned r[4] = {m, (unsigned)e, 7u, 0u};
      philox4x32_10(r, 1u, 2u);
      for (int i = 0; i < 4; ++i) {
        const float a = make(r[i] & (kMant - 1), (int)((r[i] >> 23) & 63) - 32, r[i] >> 31);
        n += !same(gen_div(a, x), __fdiv_rn(a, x));
      }
    }
  }
  if (n) atomicAdd(bad, (unsigned long long)n);
}

}  // namespace

extern "C" long long gen_arith_differences(int what, int e0, int e1) {
  unsigned long long* d = nullptr;
  unsigned long long h = 0;
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return -1;
  cudaMemset(d, 0, sizeof(h));
  const int th = 256, bl = kMant / th;
  if (what == 0) k_count<0><<<bl, th>>>(e0, e1, d);
  if (what == 1) k_count<1><<<bl, th>>>(e0, e1, d);
  if (what == 2) k_count<2><<<bl, th>>>(e0, e1, d);
  if (what == 3) k_count<3><<<bl, th>>>(e0, e1, d);
  const cudaError_t e = cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? (long long)h : -1;
}
