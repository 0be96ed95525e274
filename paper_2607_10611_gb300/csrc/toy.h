// toy.h -- launch arguments of the matrix-fitting diagnostic (internal to
// the CUDA library; the C ABI is mpadam_toy_* in include/mpadam.h).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "step_args.h"

namespace mpadam {

constexpr int kToyRunCtas = 128;  // most CTAs of a run (a power of two below the 152 SMs)
constexpr int kToyRunSteps = 8192;  // most steps of one launch

// What the CTAs of a run tell one another; all bits set when a launch starts.
struct ToySync {
  unsigned long long line[kToyRunCtas][16];  // a 128-byte line per CTA: [0] step << 32 | alpha, [1] step << 32
  unsigned long long slot[2][kToyRunCtas];   // chunk sums (binary64 bits) of even and odd steps
  uint32_t arrived[2][32];                   // per problem: CTAs that reached the barriers so far, less one
};

struct ToyArgs {
  uint16_t* w;          // [n] BF16 bits, updated in place
  const float* wstar;   // [n]
  int32_t* cnt;         // [n] hit counts (0 between steps; a run: those of its even steps)
  int32_t* first;       // [n] INT_MAX - (first sample of each entry); 0 between steps (a run: hit counts of odd steps)
  int32_t* idx;         // [batch]
  float* res;           // [batch]
  double* partial;      // [batch / 256 + 2] chunk sums of the squared residuals
  double* loss_out;     // caller's device double, or nullptr
  ToySync* sync;
  double* loss_hi;      // [kToyRunSteps] the second problem's part of each loss in a run
  int32_t* err;         // set when a run's wait gave up
  int64_t n, batch;     // powers of two; 32 <= batch / halves <= 32 * 2048
  int32_t mode, split;
  float lr_add, lr_mul, rmax, tau, c_lo, c_hi;
  uint32_t rk0[kPhiloxRounds], rk1[kPhiloxRounds];
  uint32_t t_lo, t_hi;
};

cudaError_t launch_toy_step(const ToyArgs& a, cudaStream_t stream);
// Steps first .. first + steps - 1 as cooperative launches; losses: a device
// double per step, or nullptr.
cudaError_t launch_toy_run(const ToyArgs& a, int64_t first, int64_t steps, double* losses, cudaStream_t stream);

}  // namespace mpadam
