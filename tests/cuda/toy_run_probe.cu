// Test-only build of the diagnostic's run: with REFUSE_COOPERATIVE the driver
// "refuses" every cooperative launch as too large, and MPADAM_TOY_SPIN_LIMIT
// sets how often a wait polls before it gives up.
#include <cuda_runtime.h>

#ifdef REFUSE_COOPERATIVE
static cudaError_t refuse(const void*, dim3, dim3, void**, size_t, cudaStream_t) {
  return cudaErrorCooperativeLaunchTooLarge;
}
#define cudaLaunchCooperativeKernel refuse
#endif
#include "toy.cu"

// A combined-rule run on w (device), as mpadam_toy_create and mpadam_toy_run
// set it up.  err: the device error word.  Returns a CUDA error code.
extern "C" int toy_run_probe(uint16_t* w, const float* wstar, long long n, long long batch, int split, float lr,
                             float c_lo, float c_hi, unsigned long long seed, long long first, long long steps,
                             double* losses, int* err) {
  mpadam::ToyArgs a{};
  const size_t sizes[] = {4u * (size_t)n, 4u * (size_t)n, 4u * (size_t)batch, 4u * (size_t)batch,
                          8u * ((size_t)batch / 256 + 2),
                          sizeof(mpadam::ToySync) + 8u * mpadam::kToyRunSteps + 4u};
  void* p[6] = {};
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 6 && e == cudaSuccess; ++i) {
    e = cudaMalloc(&p[i], sizes[i]);
    if (e == cudaSuccess) e = cudaMemset(p[i], 0, sizes[i]);
  }
  if (e == cudaSuccess) {
    a.w = w;
    a.wstar = wstar;
    a.cnt = (int32_t*)p[0];
    a.first = (int32_t*)p[1];
    a.idx = (int32_t*)p[2];
    a.res = (float*)p[3];
    a.partial = (double*)p[4];
    a.sync = (mpadam::ToySync*)p[5];
    a.loss_hi = (double*)(a.sync + 1);
    a.err = (int32_t*)(a.loss_hi + mpadam::kToyRunSteps);
    a.n = n;
    a.batch = batch;
    a.mode = 2;
    a.split = split;
    a.lr_add = a.lr_mul = lr;
    a.rmax = 0.75f;
    a.tau = 1e-8f;
    a.c_lo = c_lo;
    a.c_hi = split ? c_hi : c_lo;
    for (int r = 0; r < mpadam::kPhiloxRounds; ++r) {
      a.rk0[r] = (uint32_t)seed + (uint32_t)r * 0x9E3779B9u;
      a.rk1[r] = (uint32_t)(seed >> 32) + (uint32_t)r * 0xBB67AE85u;
    }
    e = mpadam::launch_toy_run(a, first, steps, losses, nullptr);
    const cudaError_t s = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = s;
    if (e == cudaSuccess) e = cudaMemcpy(err, a.err, 4, cudaMemcpyDeviceToHost);
  }
  for (void* q : p) cudaFree(q);
  return (int)e;
}
