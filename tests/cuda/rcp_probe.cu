// Test-only probe: the largest relative error of rcp.approx.ftz.f32 against
// the correctly rounded reciprocal, over caller-supplied operands whose
// reciprocals are normal.  The certified fast path assumes 2^-21.
#include <cstdint>
#include <cuda_runtime.h>

__global__ void probe(const float* b, int64_t n, float* out_rel) {
  float worst = 0.0f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b[i]));
    const float e = __frcp_rn(b[i]);
    worst = fmaxf(worst, fabsf(r - e) / e);
  }
  atomicMax(reinterpret_cast<int*>(out_rel), __float_as_int(worst));
}

extern "C" int rcp_probe(const float* b, int64_t n, float* out_rel) {
  probe<<<1024, 256>>>(b, n, out_rel);
  return (int)cudaDeviceSynchronize();
}
