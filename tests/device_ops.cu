// The quotients, reciprocals and roots of lbm_device.cuh beside CUDA's own, for
// test_gpu_device_ops.py.
#include <cuda_runtime.h>

#include "lbm_device.cuh"

using namespace lbm;
using u64 = unsigned long long;

// out[op] = largest distance in ulps from the IEEE operation, out[3 + op] = number
// of operands with any (op: a / b, 1 / b, sqrt(a))
__global__ void fp64_kernel(const double* a, const double* b, size_t n, u64* out) {
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n;
       i += size_t(gridDim.x) * blockDim.x) {
    const double got[3] = {fast_div(a[i], b[i]), recip(b[i]), fast_sqrt_pos(a[i])};
    const double want[3] = {__ddiv_rn(a[i], b[i]), __drcp_rn(b[i]), __dsqrt_rn(a[i])};
    for (int op = 0; op < 3; ++op) {
      if (isnan(got[op]) && isnan(want[op])) continue;
      const long long g = __double_as_longlong(got[op]), w = __double_as_longlong(want[op]);
      const u64 d = g > w ? u64(g) - u64(w) : u64(w) - u64(g);
      if (d == 0) continue;
      atomicMax(&out[op], d);
      atomicAdd(&out[3 + op], 1ull);
    }
  }
}

// out[op] = number of FP32 operands with bits first .. last for which the bare
// forms (kNormal) and the full ones differ (op: a / b, 1 / b, a rsqrt(a))
__global__ void fp32_kernel(unsigned first, unsigned last, u64* out) {
  u64 differ[3] = {0, 0, 0};
  for (u64 u = first + blockIdx.x * u64(blockDim.x) + threadIdx.x; u <= last;
       u += u64(gridDim.x) * blockDim.x) {
    const float b = __uint_as_float(unsigned(u));
    // a numerator of either sign from 2^-20 to 2^20, by the operand's bits
    const unsigned h = unsigned(u) * 2654435761u ^ (unsigned(u) >> 15);
    const float a = __uint_as_float((h & 0x807fffffu) | ((107u + h / 8388608u % 40u) << 23));
    differ[0] += __float_as_uint(quot<true>(a, b)) != __float_as_uint(fast_div(a, b));
    differ[1] += __float_as_uint(quot_one<true>(b, 1.f)) != __float_as_uint(fast_div(1.f, b));
    differ[2] += __float_as_uint(mul_rn(b, rsqrt_normal(b))) != __float_as_uint(fast_sqrt_pos(b));
  }
  for (int op = 0; op < 3; ++op)
    if (differ[op]) atomicAdd(&out[op], differ[op]);
}

extern "C" int fp64_ops(const double* a, const double* b, size_t n, u64* out) {
  double *da = nullptr, *db = nullptr;
  u64* d = nullptr;
  bool ok = cudaMalloc(&da, n * 8) == cudaSuccess && cudaMalloc(&db, n * 8) == cudaSuccess &&
            cudaMalloc(&d, 6 * 8) == cudaSuccess && cudaMemset(d, 0, 6 * 8) == cudaSuccess &&
            cudaMemcpy(da, a, n * 8, cudaMemcpyHostToDevice) == cudaSuccess &&
            cudaMemcpy(db, b, n * 8, cudaMemcpyHostToDevice) == cudaSuccess;
  if (ok) {
    fp64_kernel<<<608, 256>>>(da, db, n, d);
    ok = cudaGetLastError() == cudaSuccess &&
         cudaMemcpy(out, d, 6 * 8, cudaMemcpyDeviceToHost) == cudaSuccess;
  }
  cudaFree(da);
  cudaFree(db);
  cudaFree(d);
  return ok ? 0 : 1;
}

extern "C" int fp32_ops(unsigned first, unsigned last, u64* out) {
  u64* d = nullptr;
  bool ok = cudaMalloc(&d, 3 * 8) == cudaSuccess && cudaMemset(d, 0, 3 * 8) == cudaSuccess;
  if (ok) {
    fp32_kernel<<<1216, 256>>>(first, last, d);
    ok = cudaGetLastError() == cudaSuccess &&
         cudaMemcpy(out, d, 3 * 8, cudaMemcpyDeviceToHost) == cudaSuccess;
  }
  cudaFree(d);
  return ok ? 0 : 1;
}
