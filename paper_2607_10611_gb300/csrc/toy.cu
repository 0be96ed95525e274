// toy.cu -- the BF16-stored matrix-fitting diagnostic (the toy diagnostic of
// Sec. 5.1 and its appendix) on the GPU: one step samples B entries of W
// with replacement, forms the minibatch loss c (mean squared residual)^2
// (per half when the halves are separate problems), and applies the
// additive, multiplicative or combined step (no moments) to every sampled
// entry, rounding it to BF16.  The squared residuals are summed as a perfect
// binary tree of binary64 sums over adjacent samples.
//
// A single step (mpadam_toy_step) is two launches:
//   1. one CTA per aligned chunk of 256 samples draws them (Philox lanes;
//      residuals, hit counts and each entry's first sample, with atomics on
//      two n-entry scratch arrays that are zero between steps) and sums the
//      chunk's subtree: each thread draws the adjacent pair that is the
//      tree's first level;
//   2. every CTA completes the tree from the partials (at most 256 per
//      problem), forms M, the loss and alpha = 4 c M / B_h; the first sample
//      of each entry applies the entry's update (its contribution alpha r
//      added once per hit) and clears the scratch.
// A run of steps (mpadam_toy_run) is one cooperative launch that keeps its
// samples in registers from one phase to the next (toy_run_kernel).
// Every result is deterministic and equals the oracle's bit for bit.
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>

#include "step_kernel.cuh"
#include "toy.h"

namespace mpadam {
namespace {

// Sample s drawn with 32-bit lane `lane` of this step: its entry, residual,
// hit count and first-sample mark.  Returns r^2, exact in binary64.
__device__ __forceinline__ double toy_draw(const ToyArgs& a, int64_t s, uint32_t lane) {
  const int64_t Bh = a.batch / (a.split ? 2 : 1);
  const int64_t range = a.n / (a.split ? 2 : 1);
  const int64_t h = a.split ? s / Bh : 0;
  const int64_t idx = h * range + static_cast<int64_t>(static_cast<uint64_t>(lane) & static_cast<uint64_t>(range - 1));
  const float wv = __uint_as_float(static_cast<uint32_t>(a.w[idx]) << 16);
  const float r = __fsub_rn(wv, a.wstar[idx]);
  a.idx[s] = static_cast<int32_t>(idx);
  a.res[s] = r;
  atomicAdd(&a.cnt[idx], 1);
  atomicMax(&a.first[idx], INT_MAX - static_cast<int32_t>(s));  // the smallest sample wins
  return static_cast<double>(r) * static_cast<double>(r);
}

// Stage 1: CTA b of a problem draws the aligned chunk of C = min(256, B_h)
// samples [bC, bC + C) and sums their squared residuals as a perfect binary
// tree (adjacent pairs per thread, then adjacent lanes, then adjacent warps)
// into partial[problem][b].  Small chunks spread the random gathers over many
// SMs: at 65,536 samples per step, 2048-sample chunks (32 CTAs) took 14.8 us
// per step, 512 took 12.7 and 256 (256 CTAs) 12.6.
constexpr int kToyChunk = 256;
constexpr int kToyMaxPartials = 32 * 2048 / kToyChunk;  // per problem, at 65,536 samples

__global__ void __launch_bounds__(kToyChunk / 2) toy_sample_partial_kernel(const __grid_constant__ ToyArgs a) {
  __shared__ double warp_sum[32];
  const int64_t Bh = a.batch / (a.split ? 2 : 1);
  const int64_t C = Bh < kToyChunk ? Bh : kToyChunk;
  const int64_t per = Bh / C;  // chunks per problem
  const int h = static_cast<int>(blockIdx.x / per), b = static_cast<int>(blockIdx.x % per);
  const int pairs = static_cast<int>(C / 2);
  const int t = threadIdx.x;
  double x = 0.0;
  if (t < pairs) {
    // samples s and s + 1 (s even): lanes s mod 4 and s mod 4 + 1 of Philox block s / 4
    const int64_t s = h * Bh + b * C + 2 * t;
    const uint64_t blk = static_cast<uint64_t>(s) >> 2;
    const uint4 r4 = philox4x32_10(static_cast<uint32_t>(blk), static_cast<uint32_t>(blk >> 32), a.t_lo, a.t_hi,
                                   a.rk0, a.rk1);
    const bool upper = (s & 2) != 0;
    x = toy_draw(a, s, upper ? r4.z : r4.x) + toy_draw(a, s + 1, upper ? r4.w : r4.y);
  }
  const int span = pairs < 32 ? pairs : 32;  // lanes holding pair sums
  for (int off = 1; off < span; off <<= 1) {
    const double y = __shfl_xor_sync(0xFFFFFFFFu, x, off);
    x = (t & off) ? y + x : x + y;
  }
  const int nw = (pairs + 31) / 32;
  if ((t & 31) == 0 && t < pairs) warp_sum[t >> 5] = x;
  __syncthreads();
  if (t < 32) {
    double w = t < nw ? warp_sum[t] : 0.0;
    for (int off = 1; off < nw; off <<= 1) {
      const double y = __shfl_xor_sync(0xFFFFFFFFu, w, off);
      w = (t & off) ? y + w : w + y;
    }
    if (t == 0) a.partial[h * per + b] = w;
  }
}

// Stage 2 (every update CTA): the problem's partial sums, a perfect tree
// over at most 256 adjacent chunks (each lane first sums up to 8 adjacent
// ones), then M, the loss and alpha.
__device__ __forceinline__ void toy_finish_mean(const ToyArgs& a, int h, double& loss_h, float& alpha_h) {
  const int64_t Bh = a.batch / (a.split ? 2 : 1);
  const int64_t C = Bh < kToyChunk ? Bh : kToyChunk;
  const int per = static_cast<int>(Bh / C);
  const int lane = threadIdx.x & 31;
  const int q = per > 32 ? per / 32 : 1;        // adjacent partials per lane (a power of two)
  const int lanes = per > 32 ? 32 : per;        // lanes holding them
  double v[kToyMaxPartials / 32];
#pragma unroll
  for (int j = 0; j < kToyMaxPartials / 32; ++j) v[j] = j < q && lane < lanes ? a.partial[h * per + lane * q + j] : 0.0;
#pragma unroll
  for (int step = 1; step < kToyMaxPartials / 32; step <<= 1)
#pragma unroll
    for (int j = 0; j + step < kToyMaxPartials / 32; j += 2 * step)
      if (step < q) v[j] = v[j] + v[j + step];
  double w = v[0];
  for (int off = 1; off < lanes; off <<= 1) {
    const double y = __shfl_xor_sync(0xFFFFFFFFu, w, off);
    w = (lane & off) ? y + w : w + y;
  }
  const double M = w / static_cast<double>(Bh);
  const double ch = static_cast<double>(h == 0 ? a.c_lo : a.c_hi);
  loss_h = ch * M * M;
  alpha_h = static_cast<float>(((4.0 * ch) * M) / static_cast<double>(Bh));
}

// The updated BF16 weight of an entry hit k times: its contribution alpha r
// added once per hit, then the rule's plain step in binary32.
__device__ __forceinline__ uint16_t toy_updated(const ToyArgs& a, float alpha, float r, int32_t k, uint16_t wbits) {
  const float x = __fmul_rn(alpha, r);
  float g = x;
  for (int32_t i = 1; i < k; ++i) g = __fadd_rn(g, x);
  const float wf = __uint_as_float(static_cast<uint32_t>(wbits) << 16);
  const float ln2 = 0.693147180559945309417232121458f;
  const float ua = __fmul_rn(-a.lr_add, g);
  const float ge = __fmul_rn(__fmul_rn(ln2, wf), g);
  const float ut = __fmul_rn(-a.lr_mul, ge);
  const float rho = fabsf(wf) > a.tau ? fabsf(wf) : a.tau;
  float um = __fdiv_rn(ut, rho);
  um = um > a.rmax ? a.rmax : um;
  um = um < -a.rmax ? -a.rmax : um;
  float wn;
  if (a.mode == 0) wn = __fadd_rn(wf, ua);
  else if (a.mode == 1) wn = __fmaf_rn(wf, um, wf);
  else wn = __fadd_rn(__fmaf_rn(wf, um, wf), ua);
  return static_cast<uint16_t>(bf16x2_rn(wn, wn) & 0xFFFFu);
}

__global__ void toy_update_kernel(const __grid_constant__ ToyArgs a) {
  __shared__ double s_loss[2];
  __shared__ float s_alpha[2];
  const int64_t s = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  // This sample's inputs, loaded while warps 0 and 1 form the mean: the
  // entry's first-sample mark, hit count and weight are independent reads
  // (a sample that is not its entry's first uses none of them; only the first
  // writes the entry, after reading it).
  int32_t idx = 0, first = 0, k = 0;
  uint16_t wbits = 0;
  float r = 0.0f;
  if (s < a.batch) {
    idx = a.idx[s];
    first = a.first[idx];
    k = a.cnt[idx];
    wbits = a.w[idx];
    r = a.res[s];
  }
  if (threadIdx.x < 64) {  // warp 0: the first problem, warp 1: the second
    const int h = threadIdx.x >> 5;
    if (h < (a.split ? 2 : 1)) {
      double l;
      float al;
      toy_finish_mean(a, h, l, al);
      if ((threadIdx.x & 31) == 0) { s_loss[h] = l; s_alpha[h] = al; }
    }
  }
  __syncthreads();
  if (s == 0 && a.loss_out) *a.loss_out = a.split ? (0.0 + s_loss[0]) + s_loss[1] : 0.0 + s_loss[0];
  if (s >= a.batch) return;
  if (first != INT_MAX - static_cast<int32_t>(s)) return;  // the entry's first sample applies its update
  const int64_t Bh = a.batch / (a.split ? 2 : 1);
  const int h = a.split ? static_cast<int>(s / Bh) : 0;
  a.w[idx] = toy_updated(a, s_alpha[h], r, k, wbits);
  a.cnt[idx] = 0;
  a.first[idx] = 0;
}

// ---------------------------------------------------------------------------
// A run of steps as one cooperative launch.  A step moves about 2 MB and is a
// chain of dependent accesses, so what counts is what lies on that chain.  As
// two launches per step replayed from a graph it took 12.4 us per step (65,536
// samples, 16.8M entries).
//
// CTA b of G <= kToyRunCtas draws the C samples [bC, bC + C) of every step, a
// sample per thread (C = 512 and G = 128 at 65,536 samples).  The two halves
// of a split problem share nothing but the launch.
//   1. The thread reads its entry's weight and hit count; up to eight warps sum
//      the chunk's squared residuals, and the first publishes the sum in the
//      CTA's slot.  While the sums travel, every thread draws the next step's
//      sample, loads its target (constant), raises its entry's hit count in
//      the other of two count arrays and touches its weight's line: what does
//      not depend on this step's mean.  The sample that found a count at zero
//      owns the entry's update (all samples of an entry have the same
//      residual, so which one does not matter).
//   2. The problem's first CTA reads the slots, each as soon as it is no longer
//      empty, completes the tree and sends alpha to every CTA.  Owners write
//      the new weight and clear the count.
//   3. A barrier over the problem's CTAs: they count themselves in, and the
//      first CTA sends the go-ahead.  The next step's reads see every write
//      and final counts.
// Each CTA waits on a 128-byte line of its own: with every CTA polling the
// slots, a few lines of one L2 slice, a step took 8.9 us (8.0 so).  What
// bounds it now are the scattered accesses over four arrays of 235 MB together
// (weights, targets and two of hit counts) and the two exchanges: with all of
// them in L2 (1 Mi entries) a step is about a third shorter.  Slots alternate
// between two buffers, emptied by their one reader.  Publishing needs no
// fence: the slot's value depends on the reads that have to come first.
//
// binary64 runs at half a lane per cycle and scheduler here (a warp
// instruction holds the unit for 64 cycles), so the squares are formed with
// integer instructions, the sums are spread over a scheduler's worth of warps,
// and alpha takes two products on one thread.
//
// Waits are bounded: a CTA whose wait runs out sets *a.err and returns, and so
// do the others when theirs do.
// ---------------------------------------------------------------------------
#ifndef MPADAM_TOY_SPIN_LIMIT
#define MPADAM_TOY_SPIN_LIMIT (1u << 20)
#endif
constexpr uint32_t kToySpinLimit = MPADAM_TOY_SPIN_LIMIT;  // polls (about a second) before a wait gives up
constexpr unsigned long long kToyEmpty = ~0ull;  // no sum has these bits (one that would is stored as another NaN)

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// r r in binary64 (exact: 48 bits), with integer instructions for normal r.
__device__ __forceinline__ double toy_square(float r) {
  const uint32_t b = __float_as_uint(r) & 0x7FFFFFFFu;
  if (b - 0x00800000u < 0x7F000000u) {
    const uint32_t m = (b & 0x7FFFFFu) | 0x800000u;
    const uint64_t p = static_cast<uint64_t>(m) * m;  // in [2^46, 2^48)
    const uint32_t top = static_cast<uint32_t>(p >> 47);
    // biased exponent 2 (e - 127) + top + 1023; the leading bit of the shifted product adds one
    const uint64_t e = 2u * (b >> 23) + 768u + top;
    return __longlong_as_double(static_cast<long long>((e << 52) + (p << (6u - top))));
  }
  if (b == 0u) return 0.0;
  return static_cast<double>(r) * static_cast<double>(r);
}

// Perfect tree over the `n` (a power of two up to 32) lanes' values.
__device__ __forceinline__ double toy_lane_tree(double x, int n, int lane) {
  for (int off = 1; off < n; off <<= 1) {
    const double y = __shfl_xor_sync(0xFFFFFFFFu, x, off);
    x = (lane & off) ? y + x : x + y;
  }
  return x;
}

// Perfect tree over N adjacent values of one thread (in place; the sum in v[0]).
template <int N>
__device__ __forceinline__ void toy_thread_tree(double (&v)[N]) {
#pragma unroll
  for (int step = 1; step < N; step <<= 1)
#pragma unroll
    for (int j = 0; j + step < N; j += 2 * step) v[j] = v[j] + v[j + step];
}

// The perfect tree over `per` adjacent values in buf (a power of two up to
// kToyRunCtas); a warp calls it.
__device__ __forceinline__ double toy_slots_sum(int per, int lane, const double* buf) {
  constexpr int Q = kToyRunCtas / 32;
  if (per == kToyRunCtas) {
    double v[Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) v[j] = buf[lane * Q + j];
    toy_thread_tree(v);
    return toy_lane_tree(v[0], 32, lane);
  }
  if (per == 64) return toy_lane_tree(buf[2 * lane] + buf[2 * lane + 1], 32, lane);
  return toy_lane_tree(lane < per ? buf[lane] : 0.0, per, lane);
}
static_assert(kToyRunCtas == 128, "toy_slots_sum's cases");

// Waits for a problem's `per` slots, reads them into buf and sums them; a warp
// calls it.  False: gave up.
__device__ __forceinline__ bool toy_collect(const unsigned long long* slot, int per, int lane, double* buf,
                                            double& sum) {
  constexpr int Q = kToyRunCtas / 32;
  unsigned long long b[Q];
  bool ok = false;
  for (uint32_t i = 0; !ok && i < kToySpinLimit; ++i) {
    bool mine = true;
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      b[j] = lane + 32 * j < per ? ld_relaxed(&slot[lane + 32 * j]) : 0ull;
      mine = mine && b[j] != kToyEmpty;
    }
    ok = __all_sync(0xFFFFFFFFu, mine);
  }
#pragma unroll
  for (int j = 0; j < Q; ++j) buf[lane + 32 * j] = __longlong_as_double(static_cast<long long>(b[j]));
  __syncwarp();
  sum = toy_slots_sum(per, lane, buf);
  return ok;
}

// Waits until the upper half of *p is seq; the lower half in v.  False: gave up.
__device__ __forceinline__ bool toy_await(const unsigned long long* p, uint32_t seq, uint32_t& v) {
  for (uint32_t i = 0; i < kToySpinLimit; ++i) {
    const unsigned long long x = ld_relaxed(p);
    if (static_cast<uint32_t>(x >> 32) == seq) {
      v = static_cast<uint32_t>(x);
      return true;
    }
  }
  return false;
}

__global__ void __launch_bounds__(1024, 1) toy_run_kernel(const __grid_constant__ ToyArgs a, int64_t first,
                                                          int64_t steps, double* losses) {
  __shared__ __align__(16) double s_x[1024];
  __shared__ double s_w[8];
  __shared__ double s_buf[kToyRunCtas];
  __shared__ float s_alpha;
  __shared__ int s_fail;
  const int halves = a.split ? 2 : 1;
  const int64_t Bh = a.batch / halves, range = a.n / halves;
  const double inv_B = 1.0 / static_cast<double>(Bh);  // a power of two: products equal the divisions
  const int C = static_cast<int>(blockDim.x);          // a power of two, 32 to 1024
  const int per = static_cast<int>(gridDim.x) / halves;
  const int h = static_cast<int>(blockIdx.x) / per;
  const int t = static_cast<int>(threadIdx.x), lane = t & 31, warp = t >> 5;
  const int lead = h * per;  // the problem's first CTA
  const bool leader = static_cast<int>(blockIdx.x) == lead;
  const int sum_warps = C >= 128 ? C / 128 : 1;  // warps 0 .. sum_warps - 1 sum the chunk, 4 samples a lane
  const int64_t s = blockIdx.x * static_cast<int64_t>(C) + t;
  ToySync& sync = *a.sync;
  uint32_t* arrived = &sync.arrived[h][0];  // starts at ~0
  uint32_t goal = ~0u;
  if (t == 0) s_fail = 0;

  // the sample of a step: 32-bit lane s of its random bits
  auto draw = [&](int64_t step) -> int64_t {
    const uint64_t blk = static_cast<uint64_t>(s) >> 2;
    const uint64_t us = static_cast<uint64_t>(step);
    const uint4 r4 = philox4x32_10(static_cast<uint32_t>(blk), static_cast<uint32_t>(blk >> 32),
                                   static_cast<uint32_t>(us), static_cast<uint32_t>(us >> 32), a.rk0, a.rk1);
    const uint32_t q = static_cast<uint32_t>(s & 3);
    const uint32_t l = q == 0 ? r4.x : (q == 1 ? r4.y : (q == 2 ? r4.z : r4.w));
    return h * range + static_cast<int64_t>(static_cast<uint64_t>(l) & static_cast<uint64_t>(range - 1));
  };
  // the count arrays of even and odd steps (both zero between runs)
  auto count = [&](int64_t i, int64_t entry) -> int32_t* { return ((i & 1) ? a.first : a.cnt) + entry; };
  // everything before it in any CTA of the problem is seen after it by all; false: gave up
  auto barrier = [&](uint32_t seq) -> bool {
    goal += static_cast<uint32_t>(per);
    __syncthreads();
    if (t == 0) {
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrived) : "memory");
      if (!leader) {
        uint32_t v;
        if (!toy_await(&sync.line[blockIdx.x][1], seq, v)) s_fail = 1;
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
      }
    }
    if (leader && warp == 0) {
      uint32_t got = 0, spin = 0;
      do {
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(arrived) : "memory");
      } while (static_cast<int32_t>(got - goal) < 0 && ++spin < kToySpinLimit);
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
      if (static_cast<int32_t>(got - goal) < 0) s_fail = 1;
      else
        for (int c = lane; c < per; c += 32)
          st_relaxed(&sync.line[lead + c][1], static_cast<unsigned long long>(seq) << 32);
    }
    __syncthreads();
    return s_fail == 0;
  };

  int64_t idx = draw(first), idx_next = 0;
  float target = a.wstar[idx], target_next = 0.0f;
  int32_t found = atomicAdd(count(0, idx), 1), found_next = 0;  // 0: the owner
  bool ok = barrier(0u);
  for (int64_t i = 0; ok; ++i) {
    unsigned long long* slots = sync.slot[i & 1];
    const uint32_t seq = static_cast<uint32_t>(i) + 1u;
    // 1. residual and hit count (from L2: other CTAs write both)
    uint16_t wbits;
    int32_t k;
    asm volatile("ld.relaxed.gpu.global.u16 %0, [%1];" : "=h"(wbits) : "l"(a.w + idx) : "memory");
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(k) : "l"(count(i, idx)) : "memory");
    const float r = __fsub_rn(__uint_as_float(static_cast<uint32_t>(wbits) << 16), target);
    s_x[t] = toy_square(r);
    __syncthreads();
    if (warp < sum_warps) {
      double x;
      if (C >= 128) {
        const double2 p = reinterpret_cast<const double2*>(s_x)[2 * t];
        const double2 q = reinterpret_cast<const double2*>(s_x)[2 * t + 1];
        x = (p.x + p.y) + (q.x + q.y);
      } else {
        x = C == 64 ? s_x[2 * t] + s_x[2 * t + 1] : s_x[t];
      }
      x = toy_lane_tree(x, 32, lane);
      if (sum_warps > 1) {
        if (lane == 0) s_w[warp] = x;
        asm volatile("bar.sync 1, %0;" ::"r"(32 * sum_warps) : "memory");
        if (warp == 0) x = toy_lane_tree(lane < sum_warps ? s_w[lane] : 0.0, sum_warps, lane);
      }
      if (t == 0) {
        const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
        st_relaxed(&slots[blockIdx.x], b == kToyEmpty ? 0x7FF8000000000000ull : b);
      }
    }
    // the next step's sample, while the sums travel
    if (i + 1 < steps) {
      idx_next = draw(first + i + 1);
      target_next = a.wstar[idx_next];
      found_next = atomicAdd(count(i + 1, idx_next), 1);
      asm volatile("prefetch.global.L2 [%0];" ::"l"(a.w + idx_next));
    }
    // 2. the mean
    if (leader && warp == 0) {
      double sum;
      const bool got = toy_collect(slots + lead, per, lane, s_buf, sum);
      const double c_h = static_cast<double>(h == 0 ? a.c_lo : a.c_hi);
      // alpha = ((4 c) (sum / B)) / B: the powers of two only scale
      const float alpha = static_cast<float>((c_h * sum) * (4.0 * inv_B * inv_B));
      for (int c = lane; c < per; c += 32)
        if (got)
          st_relaxed(&sync.line[lead + c][0],
                     static_cast<unsigned long long>(seq) << 32 | __float_as_uint(alpha));
      if (lane == 0) {
        s_alpha = alpha;
        if (!got) s_fail = 1;
      }
    } else if (t == 0) {
      uint32_t v = 0u;
      if (!toy_await(&sync.line[blockIdx.x][0], seq, v)) s_fail = 1;
      s_alpha = __uint_as_float(v);
    }
    __syncthreads();
    if (s_fail) break;
    if (found == 0) {
      const uint16_t wn = toy_updated(a, s_alpha, r, k, wbits);
      asm volatile("st.relaxed.gpu.global.u16 [%0], %1;" ::"l"(a.w + idx), "h"(wn) : "memory");
      asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(count(i, idx)), "r"(0) : "memory");
    }
    if (leader && warp == 0) {  // empty the slots; this problem's part of the loss
      for (int c = lane; c < per; c += 32) st_relaxed(&slots[lead + c], kToyEmpty);
      if (losses) {
        const double M = toy_slots_sum(per, lane, s_buf) * inv_B;
        if (lane == 0) (h == 0 ? losses : a.loss_hi)[i] = 0.0 + static_cast<double>(h == 0 ? a.c_lo : a.c_hi) * M * M;
      }
    }
    if (i + 1 == steps) break;
    // 3. every write of this step before any read of the next
    ok = barrier(seq);
    idx = idx_next;
    target = target_next;
    found = found_next;
  }
  if (t == 0 && s_fail) atomicOr(a.err, 1);
}

// The loss of a split problem: both parts.
__global__ void toy_add_losses_kernel(double* losses, const double* hi, int64_t n) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i < n) losses[i] = losses[i] + hi[i];
}

}  // namespace

cudaError_t launch_toy_step(const ToyArgs& a, cudaStream_t stream) {
  const int halves = a.split ? 2 : 1;
  const int64_t Bh = a.batch / halves;
  const int64_t C = Bh < kToyChunk ? Bh : kToyChunk;
  toy_sample_partial_kernel<<<static_cast<unsigned>(halves * (Bh / C)), kToyChunk / 2, 0, stream>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const unsigned blocks = static_cast<unsigned>((a.batch + 255) / 256);
  toy_update_kernel<<<blocks, 256, 0, stream>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_toy_run(const ToyArgs& a, int64_t first, int64_t steps, double* losses, cudaStream_t stream) {
  const int64_t Bh = a.batch / (a.split ? 2 : 1);
  int64_t C = a.batch / kToyRunCtas;  // samples (threads) per CTA: at most 1024
  if (C < 128) C = 128;
  if (C > Bh) C = Bh;
  // a launch lasts at most some tens of milliseconds
  constexpr int64_t kMaxSteps = kToyRunSteps;
  for (int64_t done = 0; done < steps; done += kMaxSteps) {
    cudaError_t e = cudaMemsetAsync(a.sync, 0xFF, sizeof(ToySync), stream);  // empty slots, counts at ~0
    if (e != cudaSuccess) return e;
    ToyArgs args = a;
    int64_t f = first + done, n = steps - done < kMaxSteps ? steps - done : kMaxSteps;
    double* l = losses ? losses + done : nullptr;
    void* params[] = {&args, &f, &n, &l};
    e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&toy_run_kernel),
                                    dim3(static_cast<unsigned>(a.batch / C)), dim3(static_cast<unsigned>(C)), params, 0,
                                    stream);
    if (e == cudaErrorCooperativeLaunchTooLarge) {  // fewer SMs than CTAs to this process: step by step
      cudaGetLastError();
      for (int64_t i = 0; i < n; ++i) {
        args.loss_out = l ? l + i : nullptr;
        args.t_lo = static_cast<uint32_t>(static_cast<uint64_t>(f + i));
        args.t_hi = static_cast<uint32_t>(static_cast<uint64_t>(f + i) >> 32);
        if ((e = launch_toy_step(args, stream)) != cudaSuccess) return e;
      }
      continue;
    }
    if (e != cudaSuccess) return e;
    if (l && a.split) {
      toy_add_losses_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, stream>>>(l, a.loss_hi, n);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

}  // namespace mpadam
