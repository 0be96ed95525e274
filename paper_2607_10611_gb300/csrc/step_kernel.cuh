// step_kernel.cuh -- the fused M+Adam step kernel for sm_103a (GB300).
//
// One launch = one pass over every element of the tensor list.  Each CTA
// (one per SM) is a producer/consumer pipeline over its tiles:
//   - one producer warp (one elected lane) picks each tile -- the next of its
//     own range, then chunks claimed from the launch's tail pool -- posts the
//     tile and what is needed of its tensor beside the stage, and streams the
//     tile's slice of every array (weights w, gradients g and the moments mu,
//     nu, nu_e, each one contiguous run of bytes) into a multi-stage
//     shared-memory ring with 1-D TMA bulk copies (cp.async.bulk ...
//     mbarrier::complete_tx), evict-first in L2 since every byte is used once;
//     an end marker in the next stage tells the consumers that the work is done;
//   - fifteen consumer warps wait on the stage's mbarrier, read their 8
//     elements from shared memory, run the canonical binary32 update
//     (Algorithm 1 with the Algorithm 2 options, arxiv 2607.10611), round the
//     weight into its storage format (nearest-even, or stochastic with
//     Philox4x32-10 bits) and store w, mu, nu, nu_e straight back to HBM with
//     vector stores (256-bit for binary32 arrays), then release the stage.
// Memory latency is hidden by the ring, not by occupancy, so the consumers'
// instruction stream is the only other limit.  A tensor's last bytes that are
// not a whole 16-byte line, and arrays of misaligned weights or moments, are
// read by the consumers directly from global memory with the same arithmetic;
// misaligned gradients (of NVFP4 lists excepted) go through the ring all the
// same.  No tensor cores: nothing here is a contraction.
//
// Numerics: every floating-point operation of the canonical sequence is an
// explicit round-to-nearest intrinsic (__fmul_rn, __fadd_rn, __fmaf_rn,
// __fdiv_rn, __fsqrt_rn), so build flags cannot contract or approximate
// anything.  The certified fast path below uses approximate square roots and
// divisions only where a rounding test proves the stored result equal to the
// canonical one; everything else is recomputed canonically.
//
// Every wait on an mbarrier is bounded; a wait that gives up sets a bit in
// *err, the producer waits (again bounded) for its own copies in flight, and
// the CTA returns.
#pragma once

#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "step_args.h"

namespace mpadam {

constexpr uint32_t kSpinLimit = 1u << 22;  // mbarrier try_wait attempts before giving up (seconds)

// ---------------------------------------------------------------------------
// Global memory: streaming vector stores (no L1 allocation).
// ---------------------------------------------------------------------------
// 256-bit stores carry the binary32 moments (nothing else uses them), with an
// L2 evict-first policy, as measured (two or three alternating runs each):
// with it the 1.5B list ran 1.4 % faster, the ragged list, GPT-2 and the NVFP4
// regime with RNE 0.4-0.6 %, the FP8 regime 0.1 % slower, the NVFP4 regime
// with SR (0.54 B weights) 1.2 % faster, 2375 -> 2348 us.  The same hint on the
// 128-bit stores of BF16 moments slowed the 7B list by 0.2 %, so those stay
// plain.
__device__ __forceinline__ void st8(void* p, const uint32_t (&r)[8]) {
  uint64_t pol;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  asm volatile("st.global.L1::no_allocate.L2::cache_hint.v8.u32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8}, %9;"
               :
               : "l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]),
                 "r"(r[6]), "r"(r[7]), "l"(pol)
               : "memory");
}
__device__ __forceinline__ void st4(void* p, const uint32_t (&r)[4]) {
  asm volatile("st.global.L1::no_allocate.v4.u32 [%0], {%1,%2,%3,%4};"
               :
               : "l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
               : "memory");
}
__device__ __forceinline__ void st2(void* p, const uint32_t (&r)[2]) {
  asm volatile("st.global.L1::no_allocate.v2.u32 [%0], {%1,%2};"
               :
               : "l"(p), "r"(r[0]), "r"(r[1])
               : "memory");
}

// ---------------------------------------------------------------------------
// Shared memory, mbarriers and the TMA bulk copy
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void lds4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void lds2(uint32_t addr, uint32_t (&r)[2]) {
  asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t addr) {
  uint16_t h;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(h) : "r"(addr));
  return h;
}
__device__ __forceinline__ uint32_t lds_u8(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_u16(uint32_t addr, uint32_t v) {
  asm volatile("{\n .reg .b16 h;\n cvt.u16.u32 h, %1;\n st.shared.u16 [%0], h;\n}" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_u8(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u8 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Wait until the phase with the given parity has completed; false after
// kSpinLimit attempts.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (uint32_t i = 0; i < kSpinLimit; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}
__device__ __forceinline__ uint64_t evict_first_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
// 1-D bulk copy global -> shared, completing `bytes` of transaction on `bar`.
// Source and destination 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void tma_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar,
                                         uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(pol)
      : "memory");
}

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) with precomputed round
// keys rk[r] = key + r * (Weyl constants): each round takes the 64-bit
// products of words 0 and 2 with the two multipliers, feeds the high halves
// (xored with words 3 / 1 and the round key) across and the low halves
// straight through.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3,
                                               const uint32_t (&rk0)[kPhiloxRounds],
                                               const uint32_t (&rk1)[kPhiloxRounds]) {
#pragma unroll
  for (int r = 0; r < kPhiloxRounds; ++r) {
    const uint64_t pa = static_cast<uint64_t>(x0) * 0xD2511F53u;
    const uint64_t pb = static_cast<uint64_t>(x2) * 0xCD9E8D57u;
    const uint32_t y0 = static_cast<uint32_t>(pb >> 32) ^ x1 ^ rk0[r];
    const uint32_t y2 = static_cast<uint32_t>(pa >> 32) ^ x3 ^ rk1[r];
    x1 = static_cast<uint32_t>(pb);
    x3 = static_cast<uint32_t>(pa);
    x0 = y0;
    x2 = y2;
  }
  return make_uint4(x0, x1, x2, x3);
}

// ---------------------------------------------------------------------------
// The canonical per-element update.
// ---------------------------------------------------------------------------
struct Upd {
  float wn, m, v, ve;
};

template <bool OPT>
__device__ __forceinline__ Upd madam_update(const StepScalars& s, float w, float g, float m, float v,
                                            float ve) {
  Upd o;
  // additive branch (Adam moments, bias correction folded into ka and c2)
  o.m = __fmaf_rn(s.b1, m, __fmul_rn(s.omb1, g));
  o.v = __fmaf_rn(s.b2, v, __fmul_rn(s.omb2, __fmul_rn(g, g)));
  float ua = __fdiv_rn(__fmul_rn(s.ka, o.m), __fmaf_rn(__fsqrt_rn(o.v), s.c2, s.eps));
  if (OPT && s.wd_on) ua = __fsub_rn(ua, __fmul_rn(s.kwd, w));
  // multiplicative branch: exponent gradient, its second moment, proposal
  const float ge = __fmul_rn(__fmul_rn(s.ln2, w), g);
  o.ve = __fmaf_rn(s.b2, ve, __fmul_rn(s.omb2, __fmul_rn(ge, ge)));
  float n = __fdiv_rn(ge, __fmaf_rn(__fsqrt_rn(o.ve), s.c2, s.eps));
  if (OPT && s.gmax_on) n = fmaxf(-s.gmax, fminf(n, s.gmax));
  float um = __fdiv_rn(__fmul_rn(s.km, n), fmaxf(fabsf(w), s.tau));
  um = fmaxf(s.lo, fminf(um, s.hi));
  // combine: w + w u_m + u_a
  float wn = __fadd_rn(__fmaf_rn(w, um, w), ua);
  if (OPT && s.wmax_on) wn = fmaxf(-s.wmax, fminf(wn, s.wmax));
  o.wn = wn;
  return o;
}

// ---------------------------------------------------------------------------
// Packed binary32 pairs.  sm_103a multiplies and adds two binary32 values per
// instruction (f32x2), each half rounded as the scalar operation is, so a
// pair gives the same bits as two scalar operations with half the issue
// slots.  The step's instances are bound by instruction issue before they
// are by memory wherever an element has few bytes (BF16 moments, FP8 and FP4
// weights).  With the packed update, the packed encoders and the tighter
// bound below, instructions per element went from 84 to 59 (BF16 weights and
// moments, SR) and from 115 to 78 (E4M3, SR).  A 217 M-parameter list with
// BF16 moments, nearest and SR, before all this and at present: E4M3 983 ->
// 644 us and 1135 -> 822, block-scaled E4M3 991 -> 740 and 1083 -> 896, NVFP4
// 865 -> 778 and 1141 -> 946; with binary32 moments, where memory is the
// bound, NVFP4 with SR 1274 -> 1167 us and E4M3 1152 -> 1071.
// ---------------------------------------------------------------------------
using f32x2 = uint64_t;  // low half: the even element

__device__ __forceinline__ f32x2 pk(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpk(f32x2 x, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x));
}
__device__ __forceinline__ f32x2 mul2_rn(f32x2 x, f32x2 y) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ f32x2 mul2_rd(f32x2 x, f32x2 y) {
  f32x2 r;
  asm("mul.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ f32x2 mul2_ru(f32x2 x, f32x2 y) {
  f32x2 r;
  asm("mul.rp.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ f32x2 add2_rn(f32x2 x, f32x2 y) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ f32x2 add2_rd(f32x2 x, f32x2 y) {
  f32x2 r;
  asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ f32x2 fma2_rn(f32x2 x, f32x2 y, f32x2 z) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
  return r;
}

// ---------------------------------------------------------------------------
// Certified fast update (Ziv's rounding test: A. Ziv, "Fast evaluation of
// elementary mathematical functions with correctly rounded last bit", ACM
// TOMS 17(3), 1991), two elements at a time.  The moments are computed
// exactly as above; the weight update takes its two square roots from
// sqrt.approx.ftz and its three quotients as products with rcp.approx.ftz
// (the PTX manual bounds both by 2^-23 relative).
//
// With every approximate result assumed within 2^-21 relative of the exact
// one and u = 2^-24 (one rounding):
//   a denominator      fl(sqrt' c2 + eps): 2^-21 + 2u            = 1.25 2^-21
//   u_a                + reciprocal 2^-21 + 2u                   = 2.5  2^-21
//   n                  the same                                  = 2.5  2^-21
//   w u_m              + 2u (eta_m n) + reciprocal 2^-21 + 2u    = 4    2^-21
// (clamps are 1-Lipschitz and their intervals hold 0, so they keep relative
// bounds), and the two last roundings, on either side, add
// 2u (|t'| + |wn'|) <= 2u (2 |w| + 2 |w u_m'| + |u_a'|) with t = w + w u_m:
//   eps = (|w u_m'| + |u_a'|) 5 2^-21 + rho 1.25 2^-22 + 2^-96
// with rho = max(|w|, tau) >= |w|.  The constants leave a tenth to a quarter
// for second-order terms and for the roundings of eps itself.  Flushing stays
// inside these terms when eps >= 2^-28, c2 <= 2^14, eta_m <= 4 and tau >=
// 2^-125: a subnormal nu or nu_e moves its denominator by at most
// c2 2^-63 <= 2^-21 eps (in place of the square root's own 2^-21), a
// subnormal numerator or quotient moves u_a and n by at most 2^-149 / eps <=
// 2^-121 and w u_m by at most eta_m (|w| / rho) 2^-121.  A denominator is
// infinite only when its moment is (eps <= 2^60, c2 <= 2^14), and then both
// sides have a zero quotient.  The divisor rho needs no upper bound: above
// 2^126 its approximate reciprocal is flushed to 0 and the canonical
// |w u_m| <= eta_m |n| <= 4 (1 - beta2)^(-1/2) <= 2^14 (nu_e' >= (1 - beta2)
// g_e^2 bounds |n|) is far below half an ulp of w, so w + w u_m is w on both
// sides.  The host allows this path only under those conditions (cert_ok).
// wn' not finite shows as a NaN in `fin` (the product with 0), and the group
// is then recomputed.
//
// Options.  The clamps of n (g_max) and of the weight (w_max) are 1-Lipschitz
// as well; `fin` sees wn' before w_max.  With decay, u_a becomes fl(u_a -
// fl(kwd w)), kwd <= 1 (cert_ok), both sides rounding once more: at most
// 2u (|u_a| + |w|), and |wn'| grows by as much, so rho's coefficient becomes
// 2.5 2^-22 (|u_a|'s has the room).
// Before, a list with any option ran the exact sequence throughout: with
// decay and both clamps 464 M parameters in BF16 took 2188 us, now 1248 (with
// no option 1235); 217 M: E4M3, SR, binary32 moments 1663 -> 1100 us,
// block-scaled 1660 -> 1211, NVFP4 2440 -> 1294.
//
// The caller stores the encoding of wn' only when encoding wn' - eps (rounded
// down) and wn' + eps (rounded up) gives the same code: every encoder here is
// monotone, so the canonical wn, which lies in between, has that code too.
// Otherwise the element is recomputed with the exact sequence.  Results are
// therefore identical to the canonical sequence bit for bit; the test only
// decides how much work that takes.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float sqrt_approx_ftz(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx_ftz(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

struct CertPair {
  f32x2 wn;  // fast weights
  f32x2 ne;  // minus their bounds: the canonical weights lie in [wn + ne, wn - ne]
};

// m, v, ve go in as the stored moments and come back updated; `fin` collects
// wn' 0 (NaN once any wn' is not finite).
template <bool OPT>
__device__ __forceinline__ CertPair madam_cert_pair(const StepScalars& s, const StepPairs& q, float w0, float w1,
                                                    float g0, float g1, float& m0, float& m1, float& v0, float& v1,
                                                    float& e0, float& e1, f32x2& fin) {
  CertPair o;
  const f32x2 w = pk(w0, w1), g = pk(g0, g1);
  const f32x2 m = fma2_rn(q.b1, pk(m0, m1), mul2_rn(q.omb1, g));
  const f32x2 v = fma2_rn(q.b2, pk(v0, v1), mul2_rn(q.omb2, mul2_rn(g, g)));
  const f32x2 ge = mul2_rn(mul2_rn(q.ln2, w), g);
  const f32x2 ve = fma2_rn(q.b2, pk(e0, e1), mul2_rn(q.omb2, mul2_rn(ge, ge)));
  unpk(m, m0, m1);
  unpk(v, v0, v1);
  unpk(ve, e0, e1);
  float d0, d1, x0, x1;
  unpk(fma2_rn(pk(sqrt_approx_ftz(v0), sqrt_approx_ftz(v1)), q.c2, q.eps), d0, d1);
  const f32x2 ua = mul2_rn(mul2_rn(q.ka, m), pk(rcp_approx_ftz(d0), rcp_approx_ftz(d1)));
  unpk(fma2_rn(pk(sqrt_approx_ftz(e0), sqrt_approx_ftz(e1)), q.c2, q.eps), d0, d1);
  f32x2 n = mul2_rn(ge, pk(rcp_approx_ftz(d0), rcp_approx_ftz(d1)));
  if (OPT && s.gmax_on) {
    unpk(n, x0, x1);
    n = pk(fmaxf(-s.gmax, fminf(x0, s.gmax)), fmaxf(-s.gmax, fminf(x1, s.gmax)));
  }
  const float r0 = fmaxf(fabsf(w0), s.tau), r1 = fmaxf(fabsf(w1), s.tau);
  unpk(mul2_rn(mul2_rn(q.km, n), pk(rcp_approx_ftz(r0), rcp_approx_ftz(r1))), x0, x1);
  const f32x2 um = pk(fmaxf(s.lo, fminf(x0, s.hi)), fmaxf(s.lo, fminf(x1, s.hi)));
  f32x2 uad = ua;
  if (OPT && s.wd_on) uad = fma2_rn(mul2_rn(q.kwd, w), q.m1, ua);  // u_a - kwd w (the product with -1 is exact)
  o.wn = add2_rn(fma2_rn(w, um, w), uad);
  fin = fma2_rn(o.wn, 0ull, fin);
  if (OPT && s.wmax_on) {
    unpk(o.wn, x0, x1);
    o.wn = pk(fmaxf(-s.wmax, fminf(x0, s.wmax)), fmaxf(-s.wmax, fminf(x1, s.wmax)));
  }
  float a0, a1;
  unpk(mul2_rn(w, um), x0, x1);
  unpk(ua, a0, a1);
  o.ne = fma2_rn(pk(__fadd_rn(fabsf(x0), fabsf(a0)), __fadd_rn(fabsf(x1), fabsf(a1))), q.nc1,
                 fma2_rn(pk(r0, r1), q.nc2, q.nc0));
  return o;
}

// wn - ne rounded up (the product with -1 is exact).
__device__ __forceinline__ f32x2 sub2_ru(f32x2 wn, f32x2 ne, const StepPairs& q) {
  f32x2 r;
  asm("fma.rp.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(ne), "l"(q.m1), "l"(wn));
  return r;
}

// Whether any wn' collected in `fin` was not finite.
__device__ __forceinline__ bool cert_not_finite(f32x2 fin) {
  float a, b;
  unpk(fin, a, b);
  return !(a == 0.0f && b == 0.0f);
}

// The weight of the canonical sequence from the already updated (exact)
// moments: the exact fallback of the certified path.
template <bool OPT>
static __device__ __noinline__ float madam_wn_exact(const StepScalars& s, float w, float g, float m1, float v1,
                                             float ve1) {
  float ua = __fdiv_rn(__fmul_rn(s.ka, m1), __fmaf_rn(__fsqrt_rn(v1), s.c2, s.eps));
  if (OPT && s.wd_on) ua = __fsub_rn(ua, __fmul_rn(s.kwd, w));
  const float ge = __fmul_rn(__fmul_rn(s.ln2, w), g);
  float n = __fdiv_rn(ge, __fmaf_rn(__fsqrt_rn(ve1), s.c2, s.eps));
  if (OPT && s.gmax_on) n = fmaxf(-s.gmax, fminf(n, s.gmax));
  float um = __fdiv_rn(__fmul_rn(s.km, n), fmaxf(fabsf(w), s.tau));
  um = fmaxf(s.lo, fminf(um, s.hi));
  float wn = __fadd_rn(__fmaf_rn(w, um, w), ua);
  if (OPT && s.wmax_on) wn = fmaxf(-s.wmax, fminf(wn, s.wmax));
  return wn;
}

// ---------------------------------------------------------------------------
// Storage formats
// ---------------------------------------------------------------------------
__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// Two binary32 -> packed BF16 pair, nearest-even (hardware conversion).
__device__ __forceinline__ uint32_t bf16x2_rn(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

// Stochastic BF16 of x given the complement of its 16 random bits (0xFFFF -
// R): the sum carries into the kept half exactly when R < (low half of x),
// i.e. with probability (low half) / 2^16.  The result is the high half.
__device__ __forceinline__ uint32_t bf16_sr_sum(float x, uint32_t nr16) {
  const uint32_t sum = __float_as_uint(x) + nr16;
  return (x != x) ? 0x7FFF0000u : sum;
}

// E4M3 code -> binary32 (exact).
__device__ __forceinline__ float e4m3_value(uint32_t c) {
  const uint32_t mag = c & 0x7Fu;
  float val;
  if (mag >= 8u) {
    val = __uint_as_float((mag << 20) + (120u << 23));  // exponent field + 120, mantissa
  } else {
    val = __fmul_rn(__uint2float_rn(mag), 0.001953125f);  // mag * 2^-9
  }
  if (mag == 0x7Fu) val = __uint_as_float(0x7FC00000u);
  return (c & 0x80u) ? -val : val;
}

// E2M1 code (sign, 2 exponent bits with bias 1, one mantissa bit) -> binary32 (exact).
__device__ __forceinline__ float e2m1_value(uint32_t c) {
  const uint32_t mag = c & 7u;
  const uint32_t b = mag >= 2u ? ((((mag >> 1) + 126u) << 23) | ((mag & 1u) << 22)) : (mag ? 0x3F000000u : 0u);
  return __uint_as_float(b | ((c & 8u) << 28));
}

// Eight E4M3 codes (bytes of r[0], r[1], lowest byte first) -> binary32.
// E4M3 -> FP16 -> FP32 are both widening conversions, so this is exact
// (NaN codes give NaN).
__device__ __forceinline__ void e4m3x8_to_f32(const uint32_t (&r)[2], float (&x)[8]) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    uint32_t h01, h23;
    asm("{\n .reg .b16 lo, hi;\n mov.b32 {lo, hi}, %2;\n"
        " cvt.rn.f16x2.e4m3x2 %0, lo;\n cvt.rn.f16x2.e4m3x2 %1, hi;\n}"
        : "=r"(h01), "=r"(h23)
        : "r"(r[i]));
    const float2 f01 = __half22float2(*reinterpret_cast<const __half2*>(&h01));
    const float2 f23 = __half22float2(*reinterpret_cast<const __half2*>(&h23));
    x[4 * i + 0] = f01.x;
    x[4 * i + 1] = f01.y;
    x[4 * i + 2] = f23.x;
    x[4 * i + 3] = f23.y;
  }
}

// Eight bound intervals [lo, hi] (four pairs, already scaled by 2^-e, outward
// rounded) -> packed E4M3 codes (element j in byte j of ow) and the mask of
// undecided elements, whose bytes hold no code.  Magnitudes must stay below
// 512 with both ends (the caller's amax or block scale sees to it).
//
// Nearest-even: the hardware conversion of both ends, two elements each.
//
// Stochastic: a normal E4M3 code is the binary32 magnitude's top 11 bits less
// 960, one up iff r < (its low 20 bits) 2^12, i.e. iff the low 20 bits plus
// 0xFFFFF - (r >> 12) carry.  Both ends add the same K - (r >> 12), K taking
// off 960 + 9 as well, so their top 12 bits (sign, 11 bits of code - 9) are
// the codes.  An element is undecided when those differ, or when its code -
// 9 leaves [0, 128) (bits 27..30): subnormal codes, and code 8, which a
// magnitude just below 2^-6 would round to on too fine a grid, go to the
// exact encoder.  (Codes 127 and above are the caller's to rule out.)
template <bool SR>
__device__ __forceinline__ uint32_t e4m3_interval_codes(const f32x2 (&lo)[4], const f32x2 (&hi)[4],
                                                        const uint32_t (&rnd)[8], uint32_t (&ow)[2]) {
  uint32_t mask = 0u;
  if constexpr (SR) {
    constexpr uint32_t K = 0xFFFFFu - (969u << 20);
    uint32_t f[8], H[4], any = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float l0, l1, h0, h1;
      unpk(lo[i], l0, l1);
      unpk(hi[i], h0, h1);
      const uint32_t q0 = K - (rnd[2 * i] >> 12), q1 = K - (rnd[2 * i + 1] >> 12);
      const uint32_t s0 = __float_as_uint(l0) + q0, s1 = __float_as_uint(l1) + q1;
      f[2 * i] = (s0 ^ (__float_as_uint(h0) + q0)) | (s0 & 0x78000000u);
      f[2 * i + 1] = (s1 ^ (__float_as_uint(h1) + q1)) | (s1 & 0x78000000u);
      any |= f[2 * i] | f[2 * i + 1];
      H[i] = __byte_perm(s0, s1, 0x7632);  // sign | 4 bits | code - 9 | 4 bits, twice
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const uint32_t c = (__byte_perm(H[2 * i] >> 4, H[2 * i + 1] >> 4, 0x6420) & 0x7F7F7F7Fu) + 0x09090909u;
      ow[i] = c ^ (__byte_perm(H[2 * i], H[2 * i + 1], 0x7531) & 0x80808080u);
    }
    if (any >> 20) {
#pragma unroll
      for (int j = 0; j < kGroup; ++j)
        if (f[j] >> 20) mask |= 1u << j;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      uint32_t cl, ch;
      float l0, l1, l2, l3;
      unpk(lo[2 * i], l0, l1);
      unpk(lo[2 * i + 1], l2, l3);
      asm("{\n .reg .b16 a, b;\n cvt.rn.satfinite.e4m3x2.f32 a, %2, %1;\n cvt.rn.satfinite.e4m3x2.f32 b, %4, %3;\n"
          " mov.b32 %0, {a, b};\n}" : "=r"(cl) : "f"(l0), "f"(l1), "f"(l2), "f"(l3));
      unpk(hi[2 * i], l0, l1);
      unpk(hi[2 * i + 1], l2, l3);
      asm("{\n .reg .b16 a, b;\n cvt.rn.satfinite.e4m3x2.f32 a, %2, %1;\n cvt.rn.satfinite.e4m3x2.f32 b, %4, %3;\n"
          " mov.b32 %0, {a, b};\n}" : "=r"(ch) : "f"(l0), "f"(l1), "f"(l2), "f"(l3));
      ow[i] = cl;
      if (const uint32_t d = cl ^ ch) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if ((d >> (8 * j)) & 0xFFu) mask |= 1u << (4 * i + j);
      }
    }
  }
  return mask;
}

// binary32 (already scaled by 2^-e) -> E4M3 code, saturating at +-448.
template <bool SR>
__device__ __forceinline__ uint32_t e4m3_encode(float x, uint32_t r) {
  const uint32_t b = __float_as_uint(x);
  const uint32_t sign = (b >> 24) & 0x80u;
  const uint32_t a = b & 0x7FFFFFFFu;
  if (a >= 0x43E00000u) return a > 0x7F800000u ? 0x7Fu : (sign | 0x7Eu);  // NaN / >= 448
  uint32_t code;
  if (a >= 0x3C800000u) {  // |x| >= 2^-6: normal E4M3, 20 mantissa bits dropped
    const uint32_t base = (a >> 20) - 960u;
    const uint32_t rem = a & 0xFFFFFu;
    uint32_t up;
    if (SR) up = r < (rem << 12) ? 1u : 0u;
    else up = (rem > 0x80000u || (rem == 0x80000u && (base & 1u))) ? 1u : 0u;
    code = base + up;
  } else {  // subnormal E4M3: count in units of 2^-9 (scaling by 2^9 is exact)
    const float y = __fmul_rn(__uint_as_float(a), 512.0f);
    if (SR) {
      const float fl = truncf(y);
      const float frac = __fsub_rn(y, fl);  // exact
      const uint32_t thr = __float2uint_rz(__fmul_rn(frac, 4294967296.0f));
      code = __float2uint_rz(fl) + (r < thr ? 1u : 0u);
    } else {
      code = __float2uint_rn(y);  // nearest, ties to even
    }
  }
  code = code > 0x7Eu ? 0x7Eu : code;
  return sign | code;
}

// Delayed per-tensor scale: smallest e with A <= 448 * 2^e (A as binary32
// bits, finite and >= 0); keep e_cur when A = 0; clamp to [-100, 100].
__device__ __forceinline__ int32_t fp8_next_exponent(uint32_t a_bits, int32_t e_cur) {
  if (a_bits == 0u) return e_cur;
  const int32_t ef = static_cast<int32_t>(a_bits >> 23);
  int32_t k = -100;
  if (ef != 0) k = ef - 127 - 8 + ((a_bits & 0x7FFFFFu) > 0x600000u ? 1 : 0);
  return k < -100 ? -100 : (k > 100 ? 100 : k);
}

__device__ __forceinline__ float pow2f(int32_t e) {
  return __uint_as_float(static_cast<uint32_t>(e + 127) << 23);
}

// Block scales (FP16 bit patterns).  A scale written by the step is 2^k with
// k in [-24, 15]: every such power is an FP16 number (subnormal below 2^-14).
__device__ __forceinline__ uint32_t fp16_pow2_bits(int32_t k) {
  k = k < -24 ? -24 : (k > 15 ? 15 : k);
  return k >= -14 ? static_cast<uint32_t>(k + 15) << 10 : 1u << (k + 24);
}
// Value of a scale (exact widening conversion).
__device__ __forceinline__ float fp16_value(uint32_t h) {
  return __half2float(__ushort_as_half(static_cast<unsigned short>(h)));
}
// Exponent of a scale: its exponent field minus the bias for normal scales,
// floor(log2) of its subnormal value otherwise (-24 for zero); the sign is
// ignored.  Exact for the powers of two the step writes.
__device__ __forceinline__ int32_t fp16_pow2_exponent(uint32_t h) {
  const int32_t e = static_cast<int32_t>((h >> 10) & 0x1Fu);
  if (e != 0) return e - 15;
  const int32_t k = 7 - __clz(static_cast<int32_t>(h & 0x3FFu));  // floor(log2 f) - 24
  return k < -24 ? -24 : k;
}
// Block scale of the next encode: the smallest k with A <= 448 * 2^k (A as
// binary32 bits, finite and >= 0), clamped to [-24, 15]; k_old when A = 0.
// Non-decreasing in A, which the certified path relies on.
__device__ __forceinline__ int32_t block_exponent(uint32_t a_bits, int32_t k_old) {
  if (a_bits == 0u) return k_old;
  const int32_t ef = static_cast<int32_t>(a_bits >> 23);
  int32_t k = -24;
  if (ef != 0) k = ef - 127 - 8 + ((a_bits & 0x7FFFFFu) > 0x600000u ? 1 : 0);
  return k < -24 ? -24 : (k > 15 ? 15 : k);
}

__device__ __forceinline__ bool aligned(const void* p, uintptr_t bytes) {
  return (reinterpret_cast<uintptr_t>(p) & (bytes - 1)) == 0;
}

// Bytes of a tile's slice of one array that the TMA stages: the largest
// multiple of 16 within the tile, or nothing when the array's base pointer is
// not 16-byte aligned (tile starts are then misaligned too).
__device__ __forceinline__ uint32_t staged_bytes(const void* base, int count, int esize) {
  return aligned(base, 16) ? (static_cast<uint32_t>(count * esize) & ~15u) : 0u;
}

// Gradients may start anywhere and one-byte weights at any multiple of 8 (a
// reducer's bucket packs gradients without padding; a flat buffer puts tensors
// at multiples of 8 elements).  A launch with any such array runs the MIS
// instance of the kernel (read element by element, a list of 4000 ragged
// tensors in BF16 took 651 us with its gradients in a bucket, now 384; E4M3
// with BF16 moments in a flat buffer 1096, now 361).  It is an instance of its
// own because its code, though skipped for aligned arrays, slowed short
// launches by 3 to 7 % and NVFP4 with SR by 4 %; NVFP4 has none and reads them
// in the element-wise path.  Such an array keeps its place modulo 16 in its
// region of the stage, `misalign` bytes in (tiles start at multiples of 16
// bytes from the base, so that is one number per tensor); the copy covers the
// whole 16-byte lines that lie inside the array, [lo, hi) from the region's
// start (lo | hi << 16), so only a tensor's first and last group can miss
// bytes, which patch_group fills in.
__device__ __forceinline__ uint32_t misalign(const void* base) {
  return static_cast<uint32_t>(reinterpret_cast<uintptr_t>(base) & 15u);
}
__device__ __forceinline__ uint32_t staged_range(const void* base, int64_t numel, int64_t e0, int count, int esize) {
  const uintptr_t b = reinterpret_cast<uintptr_t>(base);
  if ((b & 15u) == 0u) return (static_cast<uint32_t>(count * esize) & ~15u) << 16;
  const uintptr_t a0 = b + static_cast<uintptr_t>(e0) * esize, a1 = a0 + static_cast<uintptr_t>(count) * esize;
  const uintptr_t line = a0 & ~static_cast<uintptr_t>(15);  // the region's start
  const uintptr_t first = (b + 15) & ~static_cast<uintptr_t>(15);
  const uintptr_t last = (b + static_cast<uintptr_t>(numel) * esize) & ~static_cast<uintptr_t>(15);
  const uintptr_t lo = line > first ? line : first;
  const uintptr_t up = (a1 + 15) & ~static_cast<uintptr_t>(15);
  const uintptr_t hi = up < last ? up : last;
  return hi > lo ? static_cast<uint32_t>(lo - line) | static_cast<uint32_t>(hi - line) << 16 : 0u;
}
// Whether bytes [off, off + n) of a region were copied.
__device__ __forceinline__ bool in_range(uint32_t range, uint32_t off, uint32_t n) {
  return off >= (range & 0xFFFFu) && off + n <= (range >> 16);
}

// ---------------------------------------------------------------------------
// Group loads: 8 consecutive elements from the stage.
// ---------------------------------------------------------------------------
// The same from an address that is only a multiple of the element size.
__device__ __forceinline__ void get_bf16_at(float (&x)[8], uint32_t saddr) {
  uint32_t w[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) w[i] = lds_u32((saddr & ~3u) + 4u * i);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t r = __funnelshift_r(w[i], w[i + 1], (saddr & 2u) * 8u);
    x[2 * i] = bf16_lo(r);
    x[2 * i + 1] = bf16_hi(r);
  }
}
__device__ __forceinline__ void get_f32_at(float (&x)[8], uint32_t saddr) {
#pragma unroll
  for (int j = 0; j < kGroup; ++j) x[j] = __uint_as_float(lds_u32(saddr + 4u * j));
}
__device__ __forceinline__ void get_bf16(float (&x)[8], uint32_t saddr) {
  uint32_t r[4];
  lds4(saddr, r);
#pragma unroll
  for (int i = 0; i < 4; ++i) { x[2 * i] = bf16_lo(r[i]); x[2 * i + 1] = bf16_hi(r[i]); }
}
__device__ __forceinline__ void get_f32(float (&x)[8], uint32_t saddr) {
  uint32_t a[4], b[4];
  lds4(saddr, a);
  lds4(saddr + 16, b);
#pragma unroll
  for (int i = 0; i < 4; ++i) { x[i] = __uint_as_float(a[i]); x[4 + i] = __uint_as_float(b[i]); }
}
// Eight packed E2M1 codes (element j in bits [4j, 4j + 4)) -> binary32, with
// the hardware E2M1 -> FP16 conversion (exact) and FP16 -> binary32.
__device__ __forceinline__ void e2m1x8_to_f32(uint32_t packed, float (&x)[8]) {
  uint32_t h[4];
  asm("{\n .reg .b8 b0, b1, b2, b3;\n mov.b32 {b0, b1, b2, b3}, %4;\n"
      " cvt.rn.f16x2.e2m1x2 %0, b0;\n cvt.rn.f16x2.e2m1x2 %1, b1;\n"
      " cvt.rn.f16x2.e2m1x2 %2, b2;\n cvt.rn.f16x2.e2m1x2 %3, b3;\n}"
      : "=r"(h[0]), "=r"(h[1]), "=r"(h[2]), "=r"(h[3])
      : "r"(packed));
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h[i]));
    x[2 * i] = f.x;
    x[2 * i + 1] = f.y;
  }
}

// Eight NVFP4 weights decoded with d, as one 32-bit word.
__device__ __forceinline__ void get_fp4(float (&w)[8], uint32_t saddr, float d) {
  e2m1x8_to_f32(lds_u32(saddr), w);
#pragma unroll
  for (int j = 0; j < kGroup; ++j) w[j] = __fmul_rn(w[j], d);
}
__device__ __forceinline__ void get_e4m3(float (&x)[8], uint32_t saddr, float scale) {
  uint32_t r[2];
  lds2(saddr, r);
  e4m3x8_to_f32(r, x);
#pragma unroll
  for (int j = 0; j < kGroup; ++j) x[j] = __fmul_rn(x[j], scale);
}

// Group stores (vector when whole and aligned, else element by element).  The
// single stores are volatile so that those of one array stay together and L1
// merges them by sector (217 M parameters, BF16 moments, BF16 weights 2 bytes
// off a line: 1647 -> 1507 us, 1439 with the loads below in order as well).
__device__ __forceinline__ void st_u32(void* p, uint32_t v) {
  asm volatile("st.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_u16(void* p, uint32_t v) {
  asm volatile("{\n .reg .b16 h;\n cvt.u16.u32 h, %1;\n st.global.u16 [%0], h;\n}" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_u8(void* p, uint32_t v) {
  asm volatile("st.global.u8 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void put_bf16(const uint32_t (&o)[4], void* g, int64_t e0, int valid, bool vec) {
  if (vec && valid == kGroup) {
    st4(static_cast<uint16_t*>(g) + e0, o);
  } else {
#pragma unroll
    for (int j = 0; j < kGroup; ++j)
      if (j < valid) st_u16(static_cast<uint16_t*>(g) + e0 + j, (j & 1) ? (o[j >> 1] >> 16) : (o[j >> 1] & 0xFFFFu));
  }
}
__device__ __forceinline__ void put_f32(const float (&x)[8], void* g, int64_t e0, int valid, bool vec) {
  if (vec && valid == kGroup) {
    uint32_t o[8];
#pragma unroll
    for (int j = 0; j < kGroup; ++j) o[j] = __float_as_uint(x[j]);
    st8(static_cast<float*>(g) + e0, o);
  } else {
#pragma unroll
    for (int j = 0; j < kGroup; ++j)
      if (j < valid) st_u32(static_cast<float*>(g) + e0 + j, __float_as_uint(x[j]));
  }
}
__device__ __forceinline__ void put_e4m3(const uint32_t (&o)[2], void* g, int64_t e0, int valid, bool vec) {
  if (vec && valid == kGroup) {
    st2(static_cast<uint8_t*>(g) + e0, o);
  } else {
#pragma unroll
    for (int j = 0; j < kGroup; ++j)
      if (j < valid) st_u8(static_cast<uint8_t*>(g) + e0 + j, o[j >> 2] >> (8 * (j & 3)));
  }
}

__host__ __device__ constexpr int esize_of(int dt) { return dt == kF32 ? 4 : (dt == kBF16 ? 2 : 1); }

// A tensor's table entries: from the kernel parameters when the launch
// carries them inline, else from global memory.
__device__ __forceinline__ TensorDesc desc_of(const StepArgs& a, int k) {
  return k < a.n_inline ? a.inl_desc[k] : a.desc[k];
}
__device__ __forceinline__ const void* grad_of(const StepArgs& a, int k) {
  return k < a.n_inline ? a.inl_grads[k] : a.grads[k];
}
__device__ __forceinline__ TensorAux aux_of(const StepArgs& a, int k) {
  return k < a.n_inline ? a.inl_aux[k] : a.aux[k];
}
// The tensor holding this CTA's first tile tb (which exists): scanned from
// the inline descriptors, else the host-computed table.
__device__ __forceinline__ int first_tensor(const StepArgs& a, int64_t tb) {
  if (a.n_inline == 0) return a.cta_first[blockIdx.x];
  int k = 0;
  while (k < a.n_inline - 1 && a.inl_desc[k].tile_off + (a.inl_desc[k].numel + kTile - 1) / kTile <= tb) ++k;
  return k;
}

// The tensor holding tile t, at or after tensor k (which starts at or before
// it): the last one that starts at or before t, by doubling steps and halving
// ones.  (Empty tensors start where the next one does and come before it.)
__device__ __forceinline__ int tensor_of(const StepArgs& a, int k, int64_t t) {
  auto starts = [&](int i) { return i < a.n_desc && desc_of(a, i).tile_off <= t; };
  int step = 1;
  while (starts(k + step)) { k += step; step <<= 1; }
  for (; step > 0; step >>= 1)
    if (starts(k + step)) k += step;
  return k;
}

// What the producer posts beside each stage: the tile, and everything the
// consumers need of its tensor.  The producer's loads of the tables run ahead
// by the depth of the ring; with the consumers loading them at every change of
// tensor, each of fifteen warps waited about 1.2 us for two (E4M3: three)
// dependent reads.
struct StageHead {
  void *w, *m, *v, *ve;
  const void* g;
  void* scale;       // block scales
  uint16_t* cc;      // compute copy
  int64_t goff;
  int64_t e0;        // the tile's first element
  int32_t k;         // tensor (-1: no more work)
  int32_t count;     // elements in the tile
  int32_t rot;       // the warp that takes the tile's first 256 elements (the following ones follow, cyclically)
  int32_t ring;
  float gscale;
  int32_t e_cur;     // kE4M3: this step's exponent, the maximum that sets the next one, and a lower bound
  uint32_t amax;     // of this step's maximum so far
  uint32_t seed;
  uint32_t w_range, g_range;  // what was copied of the weights (not kNVFP4) and gradients (staged_range)
};
// What the kernel holds beside the ring: the heads and two barriers per stage.
constexpr int kStaticSmem = kMaxStages * (static_cast<int>(sizeof(StageHead)) + 16);
static_assert(kStaticSmem == 1024, "no padding between them");

// The arrays that a step writes.  Each is stored by vectors when it is aligned
// itself, as each is read from the stage when it is there (load_group), so one
// array off its boundary costs its own accesses alone: 217 M parameters, BF16
// weights and gradients, binary32 moments (aligned 1152 us) with the weights 2
// bytes off a line 2644 -> 1217 us, with mu 8 bytes off 2640 -> 1230; with
// BF16 moments 2479 -> 1439 and 2598 -> 1381.
constexpr uint32_t kVecW = 1, kVecM = 2, kVecV = 4, kVecVe = 8, kVecCc = 16, kVecAll = 31;

// Per-tensor values the consumers keep while walking a tensor's tiles.
struct TensorCtx {
  TensorDesc d;        // w, m, v, ve, goff, ring
  const void* g;       // kNVFP4's exact branch (the others read gradients from the stage, or through its head)
  uint32_t gsh, wsh;   // MIS: misalign() of the gradients and of one-byte weights
  uint32_t vec;        // kVec* of the written arrays that are aligned for vector stores of whole groups
  bool fast;           // whole warps of a tile are staged, and stored with vector stores
  float dec_scale, enc_scale;
  float cc_scale;      // E4M3 per-tensor: 2^e of the new encode (compute copy)
  void* scale;         // kE4M3B (FP16) / kNVFP4 (E4M3) block scales
  uint16_t* cc;        // BF16 compute copy, or nullptr
  float gscale;        // kNVFP4 tensor scale
  float amax_seed;     // kE4M3: a lower bound of the tensor's largest exact |w'| of this step
};

template <int WD, int GD, int MD, bool MIS>
__device__ __forceinline__ void load_tensor(const StageHead& h, TensorCtx& c) {
  c.d.w = h.w;
  c.d.m = h.m;
  c.d.v = h.v;
  c.d.ve = h.ve;
  c.d.goff = h.goff;
  c.d.ring = h.ring;
  c.g = h.g;
  c.gsh = MIS ? misalign(h.g) : 0u;
  c.wsh = MIS && (WD == kE4M3 || WD == kE4M3B) ? misalign(h.w) : 0u;
  c.vec = kVecAll;
  if (!aligned(c.d.w, WD == kBF16 ? 16 : (WD == kNVFP4 ? 4 : 8))) c.vec &= ~kVecW;
  if (!aligned(c.d.m, MD == kF32 ? 32 : 16)) c.vec &= ~kVecM;
  if (!aligned(c.d.v, MD == kF32 ? 32 : 16)) c.vec &= ~kVecV;
  if (!aligned(c.d.ve, MD == kF32 ? 32 : 16)) c.vec &= ~kVecVe;
  c.fast = c.vec == kVecAll && (MIS || (aligned(c.d.w, 16) && aligned(c.g, 16)));
  c.dec_scale = c.enc_scale = c.cc_scale = 1.0f;
  c.scale = nullptr;
  c.cc = nullptr;
  c.gscale = 1.0f;
  c.amax_seed = 0.0f;
  if (WD != kBF16) {
    c.scale = h.scale;
    c.cc = h.cc;
    c.gscale = h.gscale;
    // the compute copy joins the vector path only when 16-byte aligned;
    // block scales are staged (whole tiles: 240 bytes) only when 16-byte aligned
    if (c.cc && !aligned(c.cc, 16)) { c.vec &= ~kVecCc; c.fast = false; }
    if ((WD == kE4M3B || WD == kNVFP4) && !aligned(c.scale, 16)) c.fast = false;
  }
}

// Fills in what the copies of misaligned gradients or one-byte weights left
// out of a whole group (a tensor's first or last), so that the group can be
// read from the stage.  The fence orders these writes before the next copy
// into the stage.
template <int WD, int GD>
__device__ __forceinline__ void patch_group(const StepArgs& a, const TensorCtx& x, const StageHead& h, int64_t e0,
                                            int c, uint32_t st) {
  constexpr uint32_t GS = esize_of(GD);
  const uint32_t go = x.gsh + kGroup * GS * c, wo = x.wsh + kGroup * c;
  const bool wm = (WD == kE4M3 || WD == kE4M3B) && !in_range(h.w_range, wo, kGroup);
  const bool gm = !in_range(h.g_range, go, kGroup * GS);
  if (!wm && !gm) return;
  uint32_t r[kGroup], q[kGroup];
#pragma unroll
  for (int j = 0; j < kGroup; ++j) {
    r[j] = GD == kF32 ? static_cast<const uint32_t*>(h.g)[e0 + j] : static_cast<const uint16_t*>(h.g)[e0 + j];
    if (WD == kE4M3 || WD == kE4M3B) q[j] = static_cast<const uint8_t*>(x.d.w)[e0 + j];
  }
#pragma unroll
  for (int j = 0; j < kGroup; ++j) {
    if (gm) {
      if (GD == kF32) sts_u32(st + a.off_g + go + 4u * j, r[j]);
      else sts_u16(st + a.off_g + go + 2u * j, r[j]);
    }
    if (wm) sts_u8(st + wo + j, q[j]);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// One array's eight elements of a group, each in a word of its own (a BF16 or a
// code in the low bits): from the stage when the group's bytes are there, else
// from global memory (elements from `valid` on are 0).  Those loads are volatile
// to stay in order, one array's after another's: L1, a few KB a warp beside the
// ring, holds few arrays' lines at a time.
template <int ES, bool SHIFT>
__device__ __forceinline__ void raw_group(uint32_t (&r)[8], bool staged, uint32_t saddr, const void* p, int64_t e0,
                                          int valid) {
  if (staged) {
    if (SHIFT) {
#pragma unroll
      for (int j = 0; j < kGroup; ++j)
        r[j] = ES == 4 ? lds_u32(saddr + 4u * j) : (ES == 2 ? lds_u16(saddr + 2u * j) : lds_u8(saddr + j));
    } else if (ES == 4) {
      uint32_t a[4], b[4];
      lds4(saddr, a);
      lds4(saddr + 16, b);
#pragma unroll
      for (int i = 0; i < 4; ++i) { r[i] = a[i]; r[4 + i] = b[i]; }
    } else if (ES == 2) {
      uint32_t t[4];
      lds4(saddr, t);
#pragma unroll
      for (int i = 0; i < 4; ++i) { r[2 * i] = t[i] & 0xFFFFu; r[2 * i + 1] = t[i] >> 16; }
    } else {
      uint32_t t[2];
      lds2(saddr, t);
#pragma unroll
      for (int j = 0; j < kGroup; ++j) r[j] = (t[j >> 2] >> (8 * (j & 3))) & 0xFFu;
    }
    return;
  }
  const uint8_t* q = static_cast<const uint8_t*>(p) + e0 * ES;
#pragma unroll
  for (int j = 0; j < kGroup; ++j) {
    r[j] = 0u;
    if (j < valid) {
      if (ES == 4) asm volatile("ld.global.u32 %0, [%1];" : "=r"(r[j]) : "l"(q + 4 * j) : "memory");
      else if (ES == 2) asm volatile("{\n .reg .b16 h;\n ld.global.u16 h, [%1];\n cvt.u32.u16 %0, h;\n}"
                                     : "=r"(r[j]) : "l"(q + 2 * j) : "memory");
      else asm volatile("ld.global.u8 %0, [%1];" : "=r"(r[j]) : "l"(q + j) : "memory");
    }
  }
}

// One group of a partial tile, or of a tensor whose arrays are not all staged
// or aligned: each array from the stage when it holds the whole group there,
// else element by element from global memory -- the loads of all arrays before
// the first use, so that the group waits on memory once (waiting array by
// array, a BF16-moment list of 4000 ragged tensors took 345 us, now 281).
// 8-byte loads where the alignment allows them were slower (binary32 moments,
// mu 8 bytes off: 2219 us against 1986, either with all stores single).  The
// inlined instances (binary32 moments) read a group that is wholly there in a
// block of its own: it is what a short launch's last warp runs once, and spread
// over the other branches its instructions came in too late (E4M3, 0.4 M
// parameters 8.08 -> 7.85 us).  dec: the scale the codes decode with.
template <int WD, int GD, int MD, bool MIS>
__device__ __forceinline__ void load_group(const StepArgs& a, const TensorCtx& x, const StageHead& h, int64_t e0,
                                           int count, int c, int valid, uint32_t st, float dec, float (&w)[8],
                                           float (&g)[8], float (&m)[8], float (&v)[8], float (&ve)[8]) {
  constexpr int WS = esize_of(WD), GS = esize_of(GD), MS = esize_of(MD);
  const uint32_t end = static_cast<uint32_t>(kGroup * (c + 1));  // elements through this group
  const uint32_t go = kGroup * GS * c + x.gsh, mo = kGroup * MS * c;
  const uint32_t wo = WD == kNVFP4 ? 4u * c : static_cast<uint32_t>(kGroup * WS) * c + x.wsh;
  const bool w_in = WD == kNVFP4          ? end / 2 <= staged_bytes(x.d.w, (count + 1) / 2, 1)
                    : MIS && WD != kBF16 ? in_range(h.w_range, wo, kGroup)
                                         : end * WS <= staged_bytes(x.d.w, count, WS);
  const bool g_in = MIS ? in_range(h.g_range, go, kGroup * GS) : end * GS <= staged_bytes(h.g, count, GS);
  const bool m_in = end * MS <= staged_bytes(x.d.m, count, MS), v_in = end * MS <= staged_bytes(x.d.v, count, MS);
  const bool e_in = end * MS <= staged_bytes(x.d.ve, count, MS);
  if constexpr (MD == kF32 && WD != kNVFP4) {
    if (w_in && g_in && m_in && v_in && e_in && (!MIS || WD == kBF16 || (wo & 7u) == 0u)) {
      if (WD == kBF16) get_bf16(w, st + wo);
      else get_e4m3(w, st + wo, dec);
      if (MIS && GD == kF32) get_f32_at(g, st + a.off_g + go);
      else if (MIS) get_bf16_at(g, st + a.off_g + go);
      else if (GD == kF32) get_f32(g, st + a.off_g + go);
      else get_bf16(g, st + a.off_g + go);
      get_f32(m, st + a.off_m + mo);
      get_f32(v, st + a.off_v + mo);
      get_f32(ve, st + a.off_ve + mo);
      return;
    }
  }
  uint32_t rw[8], rg[8], rm[8], rv[8], re[8];
  if (WD == kNVFP4) {  // the group's codes as the bytes of one word
    rw[0] = 0u;
    if (w_in) {
      rw[0] = lds_u32(st + wo);
    } else {
      const uint8_t* q = static_cast<const uint8_t*>(x.d.w) + (e0 >> 1);
#pragma unroll
      for (int i = 0; i < 4; ++i) rw[1 + i] = 2 * i < valid ? q[i] : 0u;
      rw[0] = rw[1] | rw[2] << 8 | rw[3] << 16 | rw[4] << 24;
    }
  } else {
    raw_group<WS, MIS && WD != kBF16>(rw, w_in, st + wo, x.d.w, e0, valid);
  }
  raw_group<GS, MIS>(rg, g_in, st + a.off_g + go, h.g, e0, valid);
  raw_group<MS, false>(rm, m_in, st + a.off_m + mo, x.d.m, e0, valid);
  raw_group<MS, false>(rv, v_in, st + a.off_v + mo, x.d.v, e0, valid);
  raw_group<MS, false>(re, e_in, st + a.off_ve + mo, x.d.ve, e0, valid);
  auto val = [](uint32_t r, int es) { return __uint_as_float(es == 4 ? r : r << 16); };
  if (WD == kNVFP4) {
    e2m1x8_to_f32(rw[0], w);
#pragma unroll
    for (int j = 0; j < kGroup; ++j) w[j] = j < valid ? __fmul_rn(w[j], dec) : 0.0f;
  } else if (WD != kBF16) {
    const uint32_t t[2] = {rw[0] | rw[1] << 8 | rw[2] << 16 | rw[3] << 24, rw[4] | rw[5] << 8 | rw[6] << 16 | rw[7] << 24};
    e4m3x8_to_f32(t, w);
#pragma unroll
    for (int j = 0; j < kGroup; ++j) w[j] = __fmul_rn(w[j], dec);
  }
#pragma unroll
  for (int j = 0; j < kGroup; ++j) {
    if (WD == kBF16) w[j] = val(rw[j], 2);
    g[j] = val(rg[j], GS);
    m[j] = val(rm[j], MS);
    v[j] = val(rv[j], MS);
    ve[j] = val(re[j], MS);
  }
}

// BF16 compute copy of eight stored E4M3 codes: code value x scale (a power
// of two, so exact), rounded to BF16 (exact as well inside BF16's range).
__device__ __forceinline__ void put_compute(const uint32_t (&codes)[2], float scale, void* cc, int64_t e0,
                                            int valid, bool vec) {
  float xd[8];
  e4m3x8_to_f32(codes, xd);
  uint32_t o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) o[i] = bf16x2_rn(__fmul_rn(xd[2 * i], scale), __fmul_rn(xd[2 * i + 1], scale));
  put_bf16(o, cc, e0, valid, vec);
}

// Whether the straight-line code of whole staged warps (TensorCtx::fast), where
// every array is aligned, goes without the tests for it and the single stores.
// As measured per instance: 217 M parameters with BF16 moments, stochastic,
// NVFP4 982 -> 953 us, block-scaled E4M3 909 -> 893; binary32 moments, 2 M
// parameters in E4M3 15.8 -> 15.4, but in BF16 8.9 -> 9.1, so not there.
template <int WD, int MD>
constexpr bool kFastStores = WD != kBF16 || MD == kBF16;

// Store the updated moments (BF16 moments nearest-even).  FAST: see kFastStores.
template <int MD, bool FAST>
__device__ __forceinline__ void put_moments(const TensorCtx& x, int64_t e0, int valid, const float (&m)[8],
                                            const float (&v)[8], const float (&ve)[8]) {
  if (MD == kF32) {
    put_f32(m, x.d.m, e0, valid, FAST || (x.vec & kVecM) != 0u);
    put_f32(v, x.d.v, e0, valid, FAST || (x.vec & kVecV) != 0u);
    put_f32(ve, x.d.ve, e0, valid, FAST || (x.vec & kVecVe) != 0u);
  } else {
    uint32_t om[4], ov[4], oe[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      om[i] = bf16x2_rn(m[2 * i], m[2 * i + 1]);
      ov[i] = bf16x2_rn(v[2 * i], v[2 * i + 1]);
      oe[i] = bf16x2_rn(ve[2 * i], ve[2 * i + 1]);
    }
    put_bf16(om, x.d.m, e0, valid, FAST || (x.vec & kVecM) != 0u);
    put_bf16(ov, x.d.v, e0, valid, FAST || (x.vec & kVecV) != 0u);
    put_bf16(oe, x.d.ve, e0, valid, FAST || (x.vec & kVecVe) != 0u);
  }
}

// Random bits of eight consecutive elements starting at global index gidx (a
// multiple of 8): 16-bit lanes (complemented, see bf16_sr_sum) for BF16
// storage, 32-bit lanes for E4M3 storage.
template <int WD>
__device__ __forceinline__ void group_random_bits(const StepArgs& a, uint64_t gidx, uint32_t (&rnd)[8]) {
  const uint64_t gi = gidx >> 3;  // global group index
  if (WD == kBF16) {
    const uint4 r = philox4x32_10(static_cast<uint32_t>(gi), static_cast<uint32_t>(gi >> 32), a.t_lo, a.t_hi,
                                  a.rk0, a.rk1);
    rnd[0] = ~r.x & 0xFFFFu; rnd[1] = ~r.x >> 16;
    rnd[2] = ~r.y & 0xFFFFu; rnd[3] = ~r.y >> 16;
    rnd[4] = ~r.z & 0xFFFFu; rnd[5] = ~r.z >> 16;
    rnd[6] = ~r.w & 0xFFFFu; rnd[7] = ~r.w >> 16;
  } else {
    const uint64_t b0 = 2ull * gi, b1 = b0 + 1ull;
    const uint4 r0 = philox4x32_10(static_cast<uint32_t>(b0), static_cast<uint32_t>(b0 >> 32), a.t_lo, a.t_hi,
                                   a.rk0, a.rk1);
    const uint4 r1 = philox4x32_10(static_cast<uint32_t>(b1), static_cast<uint32_t>(b1 >> 32), a.t_lo, a.t_hi,
                                   a.rk0, a.rk1);
    rnd[0] = r0.x; rnd[1] = r0.y; rnd[2] = r0.z; rnd[3] = r0.w;
    rnd[4] = r1.x; rnd[5] = r1.y; rnd[6] = r1.z; rnd[7] = r1.w;
  }
}

// The canonical weight of slot j of consumer c (a runtime index), from the
// original inputs in the stage at st, which must still be allocated.  dec:
// the scale its code decodes with (E4M3 formats and NVFP4).
template <int WD, int GD, int MD, bool OPT>
__device__ __forceinline__ float exact_wn_from_stage(const StepArgs& a, const TensorCtx& x, uint32_t st, int c, int j,
                                                     float dec) {
  constexpr int GS = esize_of(GD), MS = esize_of(MD);
  const uint32_t i = static_cast<uint32_t>(kGroup * c + j);
  float w;
  if constexpr (WD == kBF16) w = __uint_as_float(lds_u16(st + 2u * i) << 16);
  else if constexpr (WD == kNVFP4) w = __fmul_rn(e2m1_value((lds_u32(st + 4u * c) >> (4 * j)) & 0xFu), dec);
  else w = __fmul_rn(e4m3_value(lds_u8(st + x.wsh + i)), dec);
  auto ld = [&](uint32_t base, int es) -> float {
    return es == 4 ? __uint_as_float(lds_u32(base + 4u * i)) : __uint_as_float(lds_u16(base + 2u * i) << 16);
  };
  return madam_update<OPT>(a.s, w, ld(st + a.off_g + x.gsh, GS), ld(st + a.off_m, MS), ld(st + a.off_v, MS),
                             ld(st + a.off_ve, MS)).wn;
}

// The complemented 16-bit random lane of BF16 element j (a runtime index) of
// the group starting at global index gidx, as group_random_bits draws it.
__device__ __forceinline__ uint32_t bf16_element_random_bits(const StepArgs& a, uint64_t gidx, int j) {
  const uint64_t gi = gidx >> 3;
  const uint4 r = philox4x32_10(static_cast<uint32_t>(gi), static_cast<uint32_t>(gi >> 32), a.t_lo, a.t_hi,
                                a.rk0, a.rk1);
  const int q = j >> 1;
  const uint32_t wd = q == 0 ? r.x : (q == 1 ? r.y : (q == 2 ? r.z : r.w));
  return (j & 1) ? (~wd >> 16) : (~wd & 0xFFFFu);
}

// The 32-bit random lane of element j (a runtime index) of a group of E4M3 or
// NVFP4 weights, as group_random_bits draws it.
__device__ __forceinline__ uint32_t lane32_random_bits(const StepArgs& a, uint64_t gidx, int j) {
  const uint64_t b = (gidx >> 2) + static_cast<uint64_t>(j >> 2);
  const uint4 r = philox4x32_10(static_cast<uint32_t>(b), static_cast<uint32_t>(b >> 32), a.t_lo, a.t_hi, a.rk0,
                                a.rk1);
  const int q = j & 3;
  return q == 0 ? r.x : (q == 1 ? r.y : (q == 2 ? r.z : r.w));
}

// Update 8 loaded elements and store them (vector stores when `vec` and
// whole, else element by element).  STAGED (whole staged warps): the stage at
// st stays allocated until this returns, and the certified path's rare exact
// branch takes the undecided elements one at a time from there (c: the
// consumer), in a loop over the set bits.  Otherwise that branch uses the
// inputs held in registers.  (Measured on the 7B list: keeping the inputs
// live through the certified loop for the exact branch, 18.64 ms per step;
// this, 18.27 ms.  Reloading them from global memory was slower still, 21.6
// ms: about a tenth of the warps' groups take the branch, and each reload
// waits on DRAM while the other warps wait for its stage.)
template <int WD, int GD, int MD, bool SR, bool OPT, bool STAGED>
__device__ __forceinline__ void finish_group(const StepArgs& a, const TensorCtx& x, int64_t e0, int valid,
                                             float (&w)[8], float (&g)[8], float (&m)[8], float (&v)[8],
                                             float (&ve)[8], uint32_t& amax_bits, uint32_t st, int c) {
  // random bits: one Philox block per 8 BF16 lanes, two per 8 E4M3 lanes
  uint32_t rnd[8];
  if (SR) group_random_bits<WD>(a, static_cast<uint64_t>(x.d.goff + e0), rnd);

  if (WD == kBF16 && a.s.cert_ok) {  // certified fast path (see madam_cert_pair)
    uint32_t ow[4], df[4];  // codes of the lower ends, and where the upper ends' differ (two 16-bit halves each)
    f32x2 fin = 0ull;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const CertPair u = madam_cert_pair<OPT>(a.s, a.p, w[2 * i], w[2 * i + 1], g[2 * i], g[2 * i + 1], m[2 * i],
                                         m[2 * i + 1], v[2 * i], v[2 * i + 1], ve[2 * i], ve[2 * i + 1], fin);
      float l0, l1, h0, h1;
      unpk(add2_rd(u.wn, u.ne), l0, l1);
      unpk(sub2_ru(u.wn, u.ne, a.p), h0, h1);
      if (SR) {
        ow[i] = __byte_perm(__float_as_uint(l0) + rnd[2 * i], __float_as_uint(l1) + rnd[2 * i + 1], 0x7632);
        df[i] = ow[i] ^ __byte_perm(__float_as_uint(h0) + rnd[2 * i], __float_as_uint(h1) + rnd[2 * i + 1], 0x7632);
      } else {
        ow[i] = bf16x2_rn(l0, l1);
        df[i] = ow[i] ^ bf16x2_rn(h0, h1);
      }
    }
    if ((df[0] | df[1] | df[2] | df[3]) != 0u || cert_not_finite(fin)) {
      // rare: encode the canonical weight of the undecided elements
      uint32_t redo = cert_not_finite(fin) ? 0xFFu : 0u;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        redo |= ((df[i] & 0xFFFFu) ? 1u << (2 * i) : 0u) | ((df[i] >> 16) ? 2u << (2 * i) : 0u);
      if constexpr (STAGED) {
#pragma unroll 1
        for (uint32_t rm = redo; rm != 0u; rm &= rm - 1u) {
          const int j = __ffs(rm) - 1;
          const float xe = exact_wn_from_stage<WD, GD, MD, OPT>(a, x, st, c, j, 1.0f);
          const uint32_t code =
              SR ? (bf16_sr_sum(xe, bf16_element_random_bits(a, static_cast<uint64_t>(x.d.goff + e0), j)) >> 16)
                 : (bf16x2_rn(xe, xe) & 0xFFFFu);
          const int sh = 16 * (j & 1);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (i == (j >> 1)) ow[i] = (ow[i] & ~(0xFFFFu << sh)) | (code << sh);
        }
      } else {
#pragma unroll
        for (int j = 0; j < kGroup; ++j) {
          if ((redo >> j) & 1u) {
            const float xe = madam_wn_exact<OPT>(a.s, w[j], g[j], m[j], v[j], ve[j]);
            const uint32_t code = SR ? (bf16_sr_sum(xe, rnd[j]) >> 16) : (bf16x2_rn(xe, xe) & 0xFFFFu);
            const int sh = 16 * (j & 1);
            ow[j >> 1] = (ow[j >> 1] & ~(0xFFFFu << sh)) | (code << sh);
          }
        }
      }
    }
    put_bf16(ow, x.d.w, e0, valid, (STAGED && kFastStores<WD, MD>) || (x.vec & kVecW) != 0u);
  } else if (WD == kE4M3 && a.s.cert_ok) {
    // Certified fast path for E4M3: both ends of the bound are scaled by 2^-e
    // with outward rounding and encoded; the largest |w'| must be exact, so an
    // element whose bound may reach the threshold is recomputed as well.  The
    // threshold is the larger of this warp's running maximum and the
    // tensor's maximum flushed so far in this step: both are exact |w'| of
    // elements of this tensor, so no element below them can be the maximum.
    uint32_t ow[2];
    const float amax_f = fmaxf(__uint_as_float(amax_bits), x.amax_seed);
    f32x2 fin = 0ull, lo[4], hi[4];
    float top = 0.0f;  // the largest magnitude of any end
    const f32x2 enc = pk(x.enc_scale, x.enc_scale);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const CertPair u = madam_cert_pair<OPT>(a.s, a.p, w[2 * i], w[2 * i + 1], g[2 * i], g[2 * i + 1], m[2 * i],
                                         m[2 * i + 1], v[2 * i], v[2 * i + 1], ve[2 * i], ve[2 * i + 1], fin);
      const f32x2 l = add2_rd(u.wn, u.ne), h = sub2_ru(u.wn, u.ne, a.p);
      float l0, l1, h0, h1;
      unpk(l, l0, l1);
      unpk(h, h0, h1);
      top = fmaxf(fmaxf(top, fabsf(l0)), fabsf(h0));
      top = fmaxf(fmaxf(top, fabsf(l1)), fabsf(h1));
      lo[i] = mul2_rd(l, enc);
      hi[i] = mul2_ru(h, enc);
    }
    uint32_t redo = e4m3_interval_codes<SR>(lo, hi, rnd, ow);
    const float sat = __fmul_rn(448.0f, x.cc_scale);  // 448 2^e: from here on codes saturate
    const bool past = !(top < sat) || cert_not_finite(fin);
    const bool cand = past || top >= amax_f;
    if (STAGED ? __any_sync(0xFFFFFFFFu, cand) : cand) {
      // Maximum candidates by code: |w'| lies above the value of code - 1 and
      // below that of code + 1.  So |w'| >= amax_f has a code at or above
      // amax_f's own, rounded down, and (whole warps) the warp's largest has a
      // code at or above the warp's largest code - 1.  A warp's first group of
      // a tensor, whose threshold is still zero, recomputes a few elements
      // instead of all 256 (a 1 Mi list 13.4 -> 9.4 us, 5 M 28.5 -> 24.5).
      uint32_t cm = 0u;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const uint32_t cj = (ow[j >> 2] >> (8 * (j & 3))) & 0x7Fu;
        if (!past && !((redo >> j) & 1u)) cm = max(cm, cj);
      }
      if (STAGED) cm = __reduce_max_sync(0xFFFFFFFFu, cm);
      if (past) {
        redo = 0xFFu;
      } else if (cand) {
        const uint32_t ab = __float_as_uint(__fmul_rz(amax_f, x.enc_scale));
        const uint32_t ca = ab >= 0x3C800000u ? (ab >> 20) - 960u : 0u;
        const uint32_t least = max(ca, cm > 0u ? cm - 1u : 0u);
#pragma unroll
        for (int j = 0; j < kGroup; ++j)
          if (((ow[j >> 2] >> (8 * (j & 3))) & 0x7Fu) >= least) redo |= 1u << j;
      }
    }
    if (redo) {  // rare: the canonical weight of undecided elements and maximum candidates
      auto exact_code = [&](int j, float xe, uint32_t r) {
        const uint32_t wb = __float_as_uint(xe) & 0x7FFFFFFFu;
        if (j < valid && wb < 0x7F800000u) amax_bits = max(amax_bits, wb);
        return e4m3_encode<SR>(__fmul_rn(xe, x.enc_scale), r);
      };
      if constexpr (STAGED) {
#pragma unroll 1
        for (uint32_t rm = redo; rm != 0u; rm &= rm - 1u) {
          const int j = __ffs(rm) - 1;
          const uint32_t r = SR ? lane32_random_bits(a, static_cast<uint64_t>(x.d.goff + e0), j) : 0u;
          const uint32_t code = exact_code(j, exact_wn_from_stage<WD, GD, MD, OPT>(a, x, st, c, j, x.dec_scale), r);
          const int sh = 8 * (j & 3);
#pragma unroll
          for (int i = 0; i < 2; ++i)
            if (i == (j >> 2)) ow[i] = (ow[i] & ~(0xFFu << sh)) | (code << sh);
        }
      } else {
#pragma unroll
        for (int j = 0; j < kGroup; ++j) {
          if ((redo >> j) & 1u) {
            const uint32_t code =
                exact_code(j, madam_wn_exact<OPT>(a.s, w[j], g[j], m[j], v[j], ve[j]), SR ? rnd[j] : 0u);
            const int sh = 8 * (j & 3);
            ow[j >> 2] = (ow[j >> 2] & ~(0xFFu << sh)) | (code << sh);
          }
        }
      }
    }
    put_e4m3(ow, x.d.w, e0, valid, STAGED || (x.vec & kVecW) != 0u);
    if (x.cc) put_compute(ow, x.cc_scale, x.cc, e0, valid, STAGED || (x.vec & kVecCc) != 0u);
  } else {
  float wn[8];
#pragma unroll
  for (int j = 0; j < kGroup; ++j) {
    const Upd u = madam_update<OPT>(a.s, w[j], g[j], m[j], v[j], ve[j]);
    wn[j] = u.wn; m[j] = u.m; v[j] = u.v; ve[j] = u.ve;
  }

  if (WD == kBF16) {
    uint32_t ow[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (SR) ow[i] = __byte_perm(bf16_sr_sum(wn[2 * i], rnd[2 * i]), bf16_sr_sum(wn[2 * i + 1], rnd[2 * i + 1]), 0x7632);
      else ow[i] = bf16x2_rn(wn[2 * i], wn[2 * i + 1]);
    }
    put_bf16(ow, x.d.w, e0, valid, (STAGED && kFastStores<WD, MD>) || (x.vec & kVecW) != 0u);
  } else {
    uint32_t ow[2] = {0u, 0u};
#pragma unroll
    for (int j = 0; j < kGroup; ++j) {
      const uint32_t wb = __float_as_uint(wn[j]) & 0x7FFFFFFFu;
      if (j < valid && wb < 0x7F800000u) amax_bits = max(amax_bits, wb);
      ow[j >> 2] |= e4m3_encode<SR>(__fmul_rn(wn[j], x.enc_scale), SR ? rnd[j] : 0u) << (8 * (j & 3));
    }
    put_e4m3(ow, x.d.w, e0, valid, STAGED || (x.vec & kVecW) != 0u);
    if (x.cc) put_compute(ow, x.cc_scale, x.cc, e0, valid, STAGED || (x.vec & kVecCc) != 0u);
  }
  }
  put_moments<MD, STAGED && kFastStores<WD, MD>>(x, e0, valid, m, v, ve);
}

// One group of a partial tile, or of a tensor whose arrays are not all staged
// or aligned.  The running E4M3 maximum goes in and comes back by value: a
// reference would pin the caller's copy to local memory.
template <int WD, int GD, int MD, bool SR, bool OPT, bool MIS>
__device__ __forceinline__ uint32_t general_group(const StepArgs& a, const TensorCtx& x, const StageHead& hd,
                                                  int64_t tile_e0, int count, int c, uint32_t st,
                                                  uint32_t amax_bits) {
  if (kGroup * c >= count) return amax_bits;
  const int valid = count - kGroup * c < kGroup ? count - kGroup * c : kGroup;
  const int64_t e0 = tile_e0 + kGroup * c;
  float w[8], g[8], m[8], v[8], ve[8];
  load_group<WD, GD, MD, MIS>(a, x, hd, e0, count, c, valid, st, x.dec_scale, w, g, m, v, ve);
  finish_group<WD, GD, MD, SR, OPT, false>(a, x, e0, valid, w, g, m, v, ve, amax_bits, st, c);
  return amax_bits;
}

// The same, as a call.  Which form a kernel instance uses was measured per
// moment format.  Called, the group costs the caller a stack frame (the live
// state saved around the call), and on a short launch after an L2 flush those
// first local-memory accesses wait on DRAM: a 1 Mi-element list with
// binary32 moments ran 15.9-17.1 us called against 13.0-13.1 us inline, and
// GPT-2, the ragged list and the 1.5B list ran 0.7-1.1 % faster inline.  With
// BF16 moments the inline form slowed the whole-tile loop instead: the 7B list
// took 18.44 ms per step against 18.21 ms called (three runs each).
template <int WD, int GD, int MD, bool SR, bool OPT, bool MIS>
__device__ __noinline__ uint32_t general_group_call(const StepArgs& a, const TensorCtx& x, const StageHead& hd,
                                                    int64_t tile_e0, int count, int c, uint32_t st,
                                                    uint32_t amax_bits) {
  return general_group<WD, GD, MD, SR, OPT, MIS>(a, x, hd, tile_e0, count, c, st, amax_bits);
}

// ---------------------------------------------------------------------------
// Block-scaled E4M3 weights: the four threads of a quad hold one 32-element
// block (8 elements each).  The stored codes decode with the block's old
// scale; the block's new scale 2^k comes from the largest finite |w'| of the
// block (current scaling); the codes re-encode x = w' 2^-k.  Every lane of the
// warp must call this (the block maximum is a quad shuffle); elements j >=
// valid are padding (valid may be 0) and neither count nor get stored.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t quad_max(uint32_t x) {
  x = max(x, __shfl_xor_sync(0xFFFFFFFFu, x, 1));
  return max(x, __shfl_xor_sync(0xFFFFFFFFu, x, 2));
}

template <int GD, int MD, bool SR, bool OPT, bool STAGED>  // STAGED: see finish_group
__device__ __forceinline__ void finish_block(const StepArgs& a, const TensorCtx& x, int64_t e0, int valid,
                                             uint32_t h_old, float (&w)[8], float (&g)[8], float (&m)[8],
                                             float (&v)[8], float (&ve)[8], uint32_t st, int c) {
  uint32_t rnd[8];
  const int32_t k_old = fp16_pow2_exponent(h_old);
  const uint32_t vmask = valid >= kGroup ? 0xFFu : (valid > 0 ? (1u << valid) - 1u : 0u);
  uint32_t ow[2];
  int32_t k_new;
  if (a.s.cert_ok) {
    // Certified path (see madam_cert_pair).  Keep the fast weights and the
    // thread's largest error bound et; the block maximum then lies in
    // [max |w'| - et, max |w'| + et] (outward rounded).  When both ends give
    // the same exponent (block_exponent is monotone) that is the exact one;
    // otherwise the quad computes its exact maximum.  Each element's code is
    // then taken from its interval [w' - et, w' + et] under the new scale
    // where both ends agree, else from the exact weight.
    f32x2 wf[4], fin = 0ull;
    float nt = 0.0f, am = 0.0f;  // nt = -et
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const CertPair u = madam_cert_pair<OPT>(a.s, a.p, w[2 * i], w[2 * i + 1], g[2 * i], g[2 * i + 1], m[2 * i],
                                         m[2 * i + 1], v[2 * i], v[2 * i + 1], ve[2 * i], ve[2 * i + 1], fin);
      float x0, x1, n0, n1;
      unpk(u.wn, x0, x1);
      unpk(u.ne, n0, n1);
      wf[i] = u.wn;
      nt = fminf(fminf(nt, n0), n1);
      if (valid >= kGroup) {
        am = fmaxf(fmaxf(am, fabsf(x0)), fabsf(x1));
      } else {
        if ((vmask >> (2 * i)) & 1u) am = fmaxf(am, fabsf(x0));
        if ((vmask >> (2 * i + 1)) & 1u) am = fmaxf(am, fabsf(x1));
      }
    }
    const bool bad = cert_not_finite(fin);
    const float lo_t = bad ? 0.0f : fmaxf(__fadd_rd(am, nt), 0.0f);
    const float hi_t = bad ? INFINITY : __fsub_ru(am, nt);
    const uint32_t qlo = quad_max(__float_as_uint(lo_t));  // non-negative floats order as their bits
    const uint32_t qhi = quad_max(__float_as_uint(hi_t));
    const int32_t kl = block_exponent(qlo, k_old);
    const bool certain = qlo != 0u && qhi < 0x7E800000u /* 2^126 */ && kl == block_exponent(qhi, k_old);
    k_new = kl;
    auto exact_wn = [&](int j) -> float {
      if constexpr (STAGED) return exact_wn_from_stage<kE4M3B, GD, MD, OPT>(a, x, st, c, j, fp16_value(h_old));
      else return madam_wn_exact<OPT>(a.s, w[j], g[j], m[j], v[j], ve[j]);
    };
    if (__any_sync(0xFFFFFFFFu, !certain)) {  // exact block maximum for the undecided quads
      uint32_t amx = 0u;
      if (!certain) {
        auto take = [&](int j) {
          if ((vmask >> j) & 1u) {
            const uint32_t b = __float_as_uint(exact_wn(j)) & 0x7FFFFFFFu;
            if (b < 0x7F800000u) amx = max(amx, b);
          }
        };
        if constexpr (STAGED) {
#pragma unroll 1
          for (int j = 0; j < kGroup; ++j) take(j);
        } else {
#pragma unroll
          for (int j = 0; j < kGroup; ++j) take(j);
        }
      }
      amx = quad_max(amx);
      if (!certain) k_new = block_exponent(amx, k_old);
    }
    const float enc = pow2f(-k_new);
    const f32x2 enc2 = pk(enc, enc), nt2 = pk(nt, nt);
    f32x2 lo[4], hi[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      lo[i] = mul2_rd(add2_rd(wf[i], nt2), enc2);
      hi[i] = mul2_ru(sub2_ru(wf[i], nt2, a.p), enc2);
    }
    if (SR) group_random_bits<kE4M3B>(a, static_cast<uint64_t>(x.d.goff + e0), rnd);
    uint32_t redo = e4m3_interval_codes<SR>(lo, hi, rnd, ow);
    // past the largest scale codes saturate (448 2^15); elsewhere the scale covers the block
    if (bad || (k_new == 15 && qhi >= 0x4B600000u)) redo = 0xFFu;
    redo &= vmask;
    if (redo) {  // rare: the canonical weight of the undecided elements
      auto put = [&](int j, uint32_t r) {
        const uint32_t code = e4m3_encode<SR>(__fmul_rn(exact_wn(j), enc), r);
        const int sh = 8 * (j & 3);
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (i == (j >> 2)) ow[i] = (ow[i] & ~(0xFFu << sh)) | (code << sh);
      };
      if constexpr (STAGED) {
#pragma unroll 1
        for (uint32_t rm = redo; rm != 0u; rm &= rm - 1u) {
          const int j = __ffs(rm) - 1;
          put(j, SR ? lane32_random_bits(a, static_cast<uint64_t>(x.d.goff + e0), j) : 0u);
        }
      } else {
#pragma unroll
        for (int j = 0; j < kGroup; ++j)
          if ((redo >> j) & 1u) put(j, SR ? rnd[j] : 0u);
      }
    }
  } else {
    float wn[8];
    uint32_t amx = 0u;
#pragma unroll
    for (int j = 0; j < kGroup; ++j) {
      const Upd u = madam_update<OPT>(a.s, w[j], g[j], m[j], v[j], ve[j]);
      wn[j] = u.wn; m[j] = u.m; v[j] = u.v; ve[j] = u.ve;
      const uint32_t b = __float_as_uint(u.wn) & 0x7FFFFFFFu;
      if (((vmask >> j) & 1u) && b < 0x7F800000u) amx = max(amx, b);
    }
    k_new = block_exponent(quad_max(amx), k_old);
    const float enc = pow2f(-k_new);
    if (SR) group_random_bits<kE4M3B>(a, static_cast<uint64_t>(x.d.goff + e0), rnd);
    ow[0] = ow[1] = 0u;
#pragma unroll
    for (int j = 0; j < kGroup; ++j)
      ow[j >> 2] |= e4m3_encode<SR>(__fmul_rn(wn[j], enc), SR ? rnd[j] : 0u) << (8 * (j & 3));
  }
  put_e4m3(ow, x.d.w, e0, valid, STAGED || (x.vec & kVecW) != 0u);
  const uint32_t h_new = fp16_pow2_bits(k_new);
  if ((threadIdx.x & 3) == 0 && valid > 0) static_cast<uint16_t*>(x.scale)[e0 / kBlock] = static_cast<uint16_t>(h_new);
  if (x.cc) put_compute(ow, fp16_value(h_new), x.cc, e0, valid, STAGED || (x.vec & kVecCc) != 0u);
  put_moments<MD, STAGED>(x, e0, valid, m, v, ve);
}

// One group of a partial tile, or of a tensor whose arrays are not all
// staged: every consumer lane calls this (lanes past the tile's end with no
// elements), loading each array from the stage when its bytes were staged,
// else from global memory.
template <int GD, int MD, bool SR, bool OPT, bool MIS>
__device__ __forceinline__ void general_block_group(const StepArgs& a, const TensorCtx& x, const StageHead& hd,
                                                 int64_t tile_e0, int count,
                                                 int c, uint32_t st) {
  const int rem = count - kGroup * c;
  const int valid = rem < 0 ? 0 : (rem < kGroup ? rem : kGroup);
  const int64_t e0 = tile_e0 + kGroup * c;
  // the block's old scale: staged when the tile's scale bytes through this block were
  const int nblk = (count + kBlock - 1) / kBlock, b = c >> 2;
  uint32_t h = 0u;
  const uint16_t* sc = static_cast<const uint16_t*>(x.scale);
  if (static_cast<uint32_t>(2 * (b + 1)) <= staged_bytes(sc + tile_e0 / kBlock, nblk, 2))
    h = lds_u16(st + a.off_s + 2 * b);
  else if (b < nblk)
    h = sc[(tile_e0 / kBlock) + b];
  float w[8], g[8], m[8], v[8], ve[8];
  load_group<kE4M3B, GD, MD, MIS>(a, x, hd, e0, count, c, valid, st, fp16_value(h), w, g, m, v, ve);
  finish_block<GD, MD, SR, OPT, false>(a, x, e0, valid, h, w, g, m, v, ve, st, c);
}

// The same, as a call: with BF16 moments, as for general_group_call.  Inline,
// the FP8-regime list (block-scaled linears, binary32 moments) ran 6.02 ms per
// step against 6.08 ms called.
template <int GD, int MD, bool SR, bool OPT, bool MIS>
__device__ __noinline__ void general_block_group_call(const StepArgs& a, const TensorCtx& x, const StageHead& hd,
                                             int64_t tile_e0, int count, int c, uint32_t st) {
  general_block_group<GD, MD, SR, OPT, MIS>(a, x, hd, tile_e0, count, c, st);
}

// ---------------------------------------------------------------------------
// NVFP4 weights: E2M1 codes (OCP FP4: sign, 2 exponent bits with bias 1, one
// mantissa bit; +-{0, 0.5, 1, 1.5, 2, 3, 4, 6}), an E4M3 scale s per 16
// elements and a binary32 tensor scale G.  A weight decodes as q * d with
// d = s * G (both products rounded to binary32); a step re-encodes
// x = w' / d' (correctly rounded) under the block's new scale.  The two
// threads of a pair (lanes 2p, 2p+1) hold one block.
// ---------------------------------------------------------------------------
// binary32 -> E2M1 code: nearest-even, or stochastic (away from zero iff
// r < floor(fraction * 2^32)); |x| >= 6 and infinities saturate; NaN -> +0.
// Branch-free: with the grid spacing sp = 0.5, 1 or 2 of |x|'s binade
// ([0, 2), [2, 4), [4, 6]), q = |x| / sp (a product with the power of two
// 1 / sp: exact), its integer part k and fraction f give the code
// k + (0, 2 or 4) and the step up.
template <bool SR>
__device__ __forceinline__ uint32_t e2m1_encode(float x, uint32_t r) {
  const float a = fminf(fabsf(x), 6.0f);
  const float rsp = a < 2.0f ? 2.0f : (a < 4.0f ? 1.0f : 0.5f);
  const uint32_t off = a < 2.0f ? 0u : (a < 4.0f ? 2u : 4u);
  const float q = __fmul_rn(a, rsp);
  const float kf = truncf(q);
  const float f = __fsub_rn(q, kf);  // exact
  const uint32_t k = __float2uint_rz(kf);
  uint32_t up;
  if (SR) up = r < __float2uint_rz(__fmul_rn(f, 4294967296.0f)) ? 1u : 0u;
  else up = (f > 0.5f || (f == 0.5f && (k & 1u))) ? 1u : 0u;
  const uint32_t code = ((__float_as_uint(x) >> 28) & 8u) | (k + off + up);
  return x != x ? 0u : code;
}

// Two binary32 -> two E2M1 codes, nearest-even (hardware conversion; x0 in
// the low nibble).
__device__ __forceinline__ uint32_t e2m1x2_rn(float x0, float x1) {
  uint32_t p;
  asm("{\n .reg .b8 b;\n cvt.rn.satfinite.e2m1x2.f32 b, %2, %1;\n cvt.u32.u8 %0, b;\n}"
      : "=r"(p)
      : "f"(x0), "f"(x1));
  return p;
}

// Stochastic E2M1 code (magnitude) shared by every value of an interval of
// magnitudes [xm, xM], decided from its smaller end xm > 0 alone.  The grid
// position P(x), one unit a code, is read off binary32's own bits: over
// [1, 2), [2, 4) and [4, 6] the codes are the exponent and the top mantissa bit
// (bits 22 up, less a constant), and over [0, 1) those of 1 + x; the 22 bits
// below are the fraction, in ticks of 2^-22.  P is continuous and rises by at
// most 2^23 ticks per unit of x; 6 and above stay at P = 7.  A value steps up
// iff r < floor(frac 2^32), so its code is the integer part of P plus 2^32 - 1 -
// r in units of 2^-32; returned is s, that sum in whole ticks rounded down (1 +
// xm is too).  With ticks >= (xM - xm) 2^23 + 3 (one tick each for the rounding
// of 1 + xm, of P and of r), the sums of the whole interval lie in [s, s +
// ticks + 1 tick's remainder), so the code is s >> 22 for all of it unless
// (s ^ (s + ticks)) >> 22 is set.
// The stochastic encode is bound by issue slots, and this form converts nothing
// between binary32 and integers (three quarter-rate conversions an element
// when the integer part and fraction were taken apart): a list of 0.54 B
// weights, linear layers in NVFP4 with compute copies and binary32 moments,
// 2455 us before, 2375 after (2345 at the copy bandwidth).
__device__ __forceinline__ uint32_t e2m1_sr_ticks(float xm, uint32_t r) {
  const float a = fminf(xm, 6.0f);
  const bool sub = a < 1.0f;
  const float z = sub ? __fadd_rd(a, 1.0f) : a;
  // 2^22 - 1 less the bits of P = 0 on this side: 1.0f's for 1 + x, 0.5f's (two codes below 1.0f's) for x
  return __float_as_uint(z) + (sub ? 0x003FFFFFu - 0x3F800000u : 0x003FFFFFu - 0x3F000000u) - (r >> 10);
}

// A block scale code with the two products its covering test and the encode
// use: d = fl(v(c) G) (the block's step) and p = fl(6 d) (the largest
// magnitude the code covers: c covers A iff p >= A).
struct Fp4Code {
  uint32_t c;
  float d, p;
};

// Value of a positive finite E4M3 code (1..126) through the hardware widening
// conversion (exact: every E4M3 value is an FP16 value).
__device__ __forceinline__ float e4m3_value_cvt(uint32_t c) {
  uint32_t h;
  asm("{\n .reg .b16 lo;\n cvt.u16.u32 lo, %1;\n cvt.rn.f16x2.e4m3x2 %0, lo;\n}" : "=r"(h) : "r"(c & 0xFFu));
  return __half2float(__ushort_as_half(static_cast<unsigned short>(h & 0xFFFFu)));
}

// c in [1, 126]
__device__ __forceinline__ Fp4Code fp4_code(uint32_t c, float G) {
  Fp4Code r;
  r.c = c;
  r.d = __fmul_rn(e4m3_value_cvt(c), G);
  r.p = __fmul_rn(6.0f, r.d);
  return r;
}

// Block scale code of the next encode: the smallest code in [1, 126] that
// covers A (finite, >= 0), 126 when none does, c_old when A = 0.  Covering is
// monotone in the code, so c is that code iff c covers A and c - 1 does not
// (or c = 1).  The candidate is A / (6 G) rounded up onto the E4M3 grid;
// both tests run side by side, and only a candidate that fails them (an
// estimate within rounding of a grid point, or a step d out of the normal
// range) walks to the answer one code at a time.
static __device__ __noinline__ Fp4Code nvfp4_scale_code_walk(float A, float G, int32_t c) {
  for (int i = 0; i < 126 && c > 1 && fp4_code(static_cast<uint32_t>(c - 1), G).p >= A; ++i) --c;
  for (int i = 0; i < 126 && c < 126 && !(fp4_code(static_cast<uint32_t>(c), G).p >= A); ++i) ++c;
  return fp4_code(static_cast<uint32_t>(c), G);
}

__device__ __forceinline__ Fp4Code nvfp4_scale_code(float A, float G, uint32_t c_old) {
  if (!(A > 0.0f)) {  // the old code, whatever it holds (zero, NaN, a sign)
    Fp4Code r;
    r.c = c_old;
    r.d = __fmul_rn(e4m3_value(c_old), G);
    r.p = __fmul_rn(6.0f, r.d);
    return r;
  }
  float est;
  asm("div.approx.f32 %0, %1, %2;" : "=f"(est) : "f"(A), "f"(__fmul_rn(6.0f, G)));
  int32_t c = static_cast<int32_t>(e4m3_encode<true>(est, 0u) & 0x7Fu);  // random bits 0: rounds up
  c = c < 1 ? 1 : (c > 126 ? 126 : c);
  const Fp4Code hi = fp4_code(static_cast<uint32_t>(c), G);
  const float p_lo = c > 1 ? fp4_code(static_cast<uint32_t>(c - 1), G).p : 0.0f;
  if (hi.p >= A && (c == 1 || !(p_lo >= A))) return hi;
  return nvfp4_scale_code_walk(A, G, c);
}

// Eight packed codes (element j in bits [4j, 4j + 4)) -> the group's bytes.
__device__ __forceinline__ void put_fp4(uint32_t packed, void* w, int64_t e0, int valid, bool vec) {
  uint8_t* p = static_cast<uint8_t*>(w) + e0 / 2;
  if (vec && valid == kGroup) {
    asm volatile("st.global.L1::no_allocate.u32 [%0], %1;" ::"l"(p), "r"(packed) : "memory");
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (2 * k < valid) {
        uint32_t byte = (packed >> (8 * k)) & 0xFFu;
        if (2 * k + 1 >= valid) byte &= 0x0Fu;  // past the tensor's end: the spare nibble is 0
        p[k] = static_cast<uint8_t>(byte);
      }
    }
  }
}

__device__ __forceinline__ uint32_t pair_max(uint32_t x) {
  return max(x, __shfl_xor_sync(0xFFFFFFFFu, x, 1));
}

// One element's canonical weight recomputed from global memory after the
// stage has been released: its code (this thread overwrites it only once the
// group is done), its gradient, and the binary32 moments this thread stored
// right after the update.  Those are the values the canonical sequence feeds
// into the weight update, so this serves binary32 moments only (BF16 moments
// are stored rounded).  L2-only loads: the moments were written by this
// thread.  Out of line: the call is rare and its pointers would otherwise stay
// live through the encode.
template <int GD, bool OPT>
__device__ __noinline__ float fp4_exact_from_global(const StepArgs& a, const TensorCtx& x, int64_t e,
                                                    float d_old) {
  const uint8_t* pw = static_cast<const uint8_t*>(x.d.w) + (e >> 1);
  uint32_t byte, bg, bm, bv, be;
  asm volatile("ld.global.cg.u8 %0, [%1];" : "=r"(byte) : "l"(pw) : "memory");
  const float w = __fmul_rn(e2m1_value((e & 1) ? (byte >> 4) : (byte & 0xFu)), d_old);
  if (GD == kF32) {
    asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(bg) : "l"(static_cast<const float*>(x.g) + e) : "memory");
  } else {
    asm volatile("ld.global.cg.u16 %0, [%1];" : "=r"(bg) : "l"(static_cast<const uint16_t*>(x.g) + e) : "memory");
    bg <<= 16;
  }
  asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(bm) : "l"(static_cast<const float*>(x.d.m) + e) : "memory");
  asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(bv) : "l"(static_cast<const float*>(x.d.v) + e) : "memory");
  asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(be) : "l"(static_cast<const float*>(x.d.ve) + e) : "memory");
  return madam_wn_exact<OPT>(a.s, w, __uint_as_float(bg), __uint_as_float(bm), __uint_as_float(bv), __uint_as_float(be));
}

// Where the rare exact branch of finish_fp4 finds an element's inputs:
// kExactRegs -- still in registers (the moments are stored at the end);
// kExactStage -- in the stage at `st` (thread c), kept until the group is done;
// kExactGlobal -- in global memory (binary32 moments only; the stage has
// already been released).  The last two store the new moments right after
// the update, so fewer values live in registers through the encode.
constexpr int kExactRegs = 0, kExactStage = 1, kExactGlobal = 2;

template <int GD, int MD, bool SR, bool OPT, int SRC>
__device__ __forceinline__ void finish_fp4(const StepArgs& a, const TensorCtx& x, int64_t e0, int valid,
                                           uint32_t c_old, float (&w)[8], float (&g)[8], float (&m)[8],
                                           float (&v)[8], float (&ve)[8], uint32_t st, int c) {
  const float G = x.gscale;
  const float d_old = __fmul_rn(e4m3_value(c_old), G);
  const uint64_t gi = static_cast<uint64_t>(x.d.goff + e0) >> 3;  // global group index (random lanes)
  const uint32_t vmask = valid >= kGroup ? 0xFFu : (valid > 0 ? (1u << valid) - 1u : 0u);
  uint32_t packed = 0u;  // element j's code in bits [4j, 4j + 4)
  uint32_t c_new;
  float d;
  static_assert(SRC != kExactGlobal || MD == kF32, "exact recompute from global needs binary32 moments");
  auto exact_wn = [&](int j) -> float {
    if constexpr (SRC == kExactStage) return exact_wn_from_stage<kNVFP4, GD, MD, OPT>(a, x, st, c, j, d_old);
    else if constexpr (SRC == kExactGlobal) return fp4_exact_from_global<GD, OPT>(a, x, e0 + j, d_old);
    else return madam_wn_exact<OPT>(a.s, w[j], g[j], m[j], v[j], ve[j]);
  };
  if (a.s.cert_ok) {
    // Certified path, as for block-scaled E4M3: fast weights and one error
    // bound et; the pair's maximum bounds decide the scale code (exact
    // maximum where they do not); then each element's interval, divided by
    // d through an approximate reciprocal, is encoded at both ends.
    float wf[8];
    float nt = 0.0f, am = 0.0f;
    f32x2 fin = 0ull;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const CertPair u = madam_cert_pair<OPT>(a.s, a.p, w[2 * i], w[2 * i + 1], g[2 * i], g[2 * i + 1], m[2 * i],
                                         m[2 * i + 1], v[2 * i], v[2 * i + 1], ve[2 * i], ve[2 * i + 1], fin);
      float n0, n1;
      unpk(u.wn, wf[2 * i], wf[2 * i + 1]);
      unpk(u.ne, n0, n1);
      nt = fminf(fminf(nt, n0), n1);
      if (valid >= kGroup) {
        am = fmaxf(fmaxf(am, fabsf(wf[2 * i])), fabsf(wf[2 * i + 1]));
      } else {
        if ((vmask >> (2 * i)) & 1u) am = fmaxf(am, fabsf(wf[2 * i]));
        if ((vmask >> (2 * i + 1)) & 1u) am = fmaxf(am, fabsf(wf[2 * i + 1]));
      }
    }
    if constexpr (SRC != kExactRegs) put_moments<MD, true>(x, e0, valid, m, v, ve);
    const float et = -nt;
    const uint32_t bad = cert_not_finite(fin) ? vmask : 0u;
    const float lo_t = bad ? 0.0f : fmaxf(__fsub_rd(am, et), 0.0f);
    const float hi_t = bad ? INFINITY : __fadd_ru(am, et);
    const uint32_t plo = pair_max(__float_as_uint(lo_t));
    const uint32_t phi = pair_max(__float_as_uint(hi_t));
    const Fp4Code cl = nvfp4_scale_code(__uint_as_float(plo), G, c_old);
    // the upper bound has the same code iff that code still covers it (or is the top one)
    const bool certain = plo != 0u && phi < 0x7E800000u /* 2^126 */ &&
                         (cl.c == 126u || cl.p >= __uint_as_float(phi));
    Fp4Code cn = cl;
    if (__any_sync(0xFFFFFFFFu, !certain)) {  // exact block maximum for the undecided pairs
      uint32_t amx = 0u;
      if (!certain) {
#pragma unroll
        for (int j = 0; j < kGroup; ++j) {
          if ((vmask >> j) & 1u) {
            const uint32_t bb = __float_as_uint(exact_wn(j)) & 0x7FFFFFFFu;
            if (bb < 0x7F800000u) amx = max(amx, bb);
          }
        }
      }
      amx = pair_max(amx);
      if (!certain) cn = nvfp4_scale_code(__uint_as_float(amx), G, c_old);
    }
    c_new = cn.c;
    d = __fmul_rn(e4m3_value(c_new), G);  // = cn.d, recomputed: fewer values live across the branch
    uint32_t redo = bad;
    if (d >= 1.1754943508222875e-38f /* 2^-126 */ && d <= 8.507059173023462e+37f /* 2^126 */) {
      // w' / d for w' in [wf - et, wf + et]: q = wf * inv (inv = rcp.approx(d),
      // 1 ulp; the product half an ulp) is within 2^-22 |q| of wf / d, and
      // et / d <= et inv (1 + 2^-22); widened to 2^-20 and 2^-126 absolute.
      float inv;
      asm("rcp.approx.f32 %0, %1;" : "=f"(inv) : "f"(d));
      const float ei = __fmaf_ru(et, __fmul_ru(inv, 1.0000009536743164f /* 1 + 2^-20 */), 1.1754943508222875e-38f);
      auto ends = [&](int j, float& xl, float& xh) {
        const float q = __fmul_rn(wf[j], inv);
        const float e2 = __fmaf_ru(fabsf(q), 9.5367431640625e-07f /* 2^-20 */, ei);
        xl = __fsub_rd(q, e2);
        xh = __fadd_ru(q, e2);
      };
      if (SR) {
        uint32_t rnd[8];
        group_random_bits<kNVFP4>(a, gi << 3, rnd);
        // The group's ticks.  An interval's magnitudes span xM - xm <= 3.5 e2:
        // 2 e2 from ends() (e2 its bound), one directed rounding at each end
        // (each within e2 / 8, since e2 >= |q| 2^-20) and the lower end below
        // taken |q| 2^-20 lower still.  With e2 <= (8 2^-20 + ei)(1 + 2^-23)
        // while |q| <= 8, (xM - xm) 2^23 + 3 <= 2^8 + ei 2^25 + 3.  Larger |q|
        // saturates at both ends; from ei = 2^-3 on nothing is certified
        // (2^22 ticks always reach the next code).
        const uint32_t ticks =
            ei <= 5.9604644775390625e-08f /* 2^-24 */
                ? 264u
                : __float2uint_ru(fminf(__fmaf_ru(ei, 33554432.0f /* 2^25 */, 260.0f), 4194304.0f /* 2^22 */));
        const float inv_lo = __fmul_rd(inv, 0.999998092651367188f /* 1 - 2^-19 */);
        // a lower bound of the smaller magnitude of ends(): |wf| inv (1 - 2^-19)
        // (below |q| (1 - 2^-20), q = wf inv rounded) less ei, rounded down
        auto low_end = [&](int j) { return __fmaf_rd(fabsf(wf[j]), inv_lo, -ei); };
        uint32_t cross = 0u;
        float xmin = INFINITY;
#pragma unroll
        for (int j = 0; j < kGroup; ++j) {
          const float xm = low_end(j);
          const uint32_t s = e2m1_sr_ticks(xm, rnd[j]);
          cross |= s ^ (s + ticks);
          xmin = fminf(xmin, xm);
          const uint32_t sign = __float_as_uint(wf[j]) >> 31;
          packed |= ((s >> 22) & 7u) << (4 * j) | sign << (4 * j + 3);
        }
        if ((cross >> 22) || !(xmin > 0.0f)) {  // rare: which elements
#pragma unroll
          for (int j = 0; j < kGroup; ++j) {
            const float xm = low_end(j);
            const uint32_t s = e2m1_sr_ticks(xm, rnd[j]);
            if (((s ^ (s + ticks)) >> 22) || !(xm > 0.0f)) redo |= 1u << j;
          }
        }
      } else {  // two elements at a time, both ends
        uint32_t diff = 0u;
#pragma unroll
        for (int i = 0; i < kGroup / 2; ++i) {
          float l0, h0, l1, h1;
          ends(2 * i, l0, h0);
          ends(2 * i + 1, l1, h1);
          const uint32_t bl = e2m1x2_rn(l0, l1);
          packed |= bl << (8 * i);
          diff |= (bl ^ e2m1x2_rn(h0, h1)) << (8 * i);
        }
#pragma unroll
        for (int j = 0; j < kGroup; ++j)
          if ((diff >> (4 * j)) & 0xFu) redo |= 1u << j;
      }
    } else {
      redo = 0xFFu;
    }
    redo &= vmask;
    if (redo) {  // rare: the canonical weight of the undecided elements
      uint32_t rnd[8];
      if (SR) group_random_bits<kNVFP4>(a, gi << 3, rnd);
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        if ((redo >> j) & 1u) {
          const float xe = __fdiv_rn(exact_wn(j), d);
          packed = (packed & ~(0xFu << (4 * j))) | ((e2m1_encode<SR>(xe, SR ? rnd[j] : 0u) & 0xFu) << (4 * j));
        }
      }
    }
    if constexpr (SRC == kExactRegs) put_moments<MD, false>(x, e0, valid, m, v, ve);
  } else {
    float wn[8];
    uint32_t amx = 0u;
#pragma unroll
    for (int j = 0; j < kGroup; ++j) {
      const Upd u = madam_update<OPT>(a.s, w[j], g[j], m[j], v[j], ve[j]);
      wn[j] = u.wn; m[j] = u.m; v[j] = u.v; ve[j] = u.ve;
      const uint32_t bb = __float_as_uint(u.wn) & 0x7FFFFFFFu;
      if (((vmask >> j) & 1u) && bb < 0x7F800000u) amx = max(amx, bb);
    }
    const Fp4Code cn = nvfp4_scale_code(__uint_as_float(pair_max(amx)), G, c_old);
    c_new = cn.c;
    d = cn.d;
    uint32_t rnd[8];
    if (SR) group_random_bits<kNVFP4>(a, gi << 3, rnd);
#pragma unroll
    for (int j = 0; j < kGroup; ++j)
      packed |= (e2m1_encode<SR>(__fdiv_rn(wn[j], d), SR ? rnd[j] : 0u) & 0xFu) << (4 * j);
    put_moments<MD, SRC != kExactRegs>(x, e0, valid, m, v, ve);
  }
  put_fp4(packed, x.d.w, e0, valid, SRC != kExactRegs || (x.vec & kVecW) != 0u);
  if ((threadIdx.x & 1) == 0 && valid > 0) static_cast<uint8_t*>(x.scale)[e0 / kFp4Block] = static_cast<uint8_t>(c_new);
  if (x.cc) {
    float q[8];
    e2m1x8_to_f32(packed, q);
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = bf16x2_rn(__fmul_rn(q[2 * i], d), __fmul_rn(q[2 * i + 1], d));
    put_bf16(o, x.cc, e0, valid, SRC != kExactRegs || (x.vec & kVecCc) != 0u);
  }
}

// One NVFP4 group of a partial tile or of a tensor whose arrays are not all
// staged; every consumer lane calls this (the block maximum is a pair shuffle).
template <int GD, int MD, bool SR, bool OPT>
__device__ __noinline__ void general_fp4_group(const StepArgs& a, const TensorCtx& x, const StageHead& hd,
                                               int64_t tile_e0, int count,
                                               int c, uint32_t st) {
  const int rem = count - kGroup * c;
  const int valid = rem < 0 ? 0 : (rem < kGroup ? rem : kGroup);
  const int64_t e0 = tile_e0 + kGroup * c;
  const int nblk = (count + kFp4Block - 1) / kFp4Block, b = c >> 1;
  const uint8_t* sc = static_cast<const uint8_t*>(x.scale);
  uint32_t s_old = 0u;
  if (static_cast<uint32_t>(b + 1) <= staged_bytes(sc + tile_e0 / kFp4Block, nblk, 1))
    s_old = lds_u8(st + a.off_s + b);
  else if (b < nblk)
    s_old = sc[(tile_e0 / kFp4Block) + b];
  const float d_old = __fmul_rn(e4m3_value(s_old), x.gscale);
  float w[8], g[8], m[8], v[8], ve[8];
  load_group<kNVFP4, GD, MD, false>(a, x, hd, e0, count, c, valid, st, d_old, w, g, m, v, ve);
  finish_fp4<GD, MD, SR, OPT, kExactRegs>(a, x, e0, valid, s_old, w, g, m, v, ve, st, c);
}

// ---------------------------------------------------------------------------
// The step kernel.
// ---------------------------------------------------------------------------
template <int WD, int GD, int MD, bool SR, bool OPT, bool MIS>
__global__ void __launch_bounds__(kThreads, 1) step_kernel(const __grid_constant__ StepArgs a) {
  constexpr int WS = esize_of(WD), GS = esize_of(GD), MS = esize_of(MD);
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages];
  __shared__ __align__(8) uint64_t empty_bar[kMaxStages];
  __shared__ StageHead heads[kMaxStages];

  // Programmatic dependent launch: the next launch of the stream may start its
  // own entry (it waits below, like this one, for everything before it).
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int S = a.stages;
  const int64_t T = a.total_tiles;
  const bool pooled = a.pool_chunks > 0;
  const int64_t split = a.pool_len > 0 ? a.pool_base - a.tile_base : T;  // tiles dealt out to the CTAs' ranges
  const int64_t tb = a.tile_base + static_cast<int64_t>(blockIdx.x) * split / gridDim.x;
  const int64_t te = a.tile_base + (static_cast<int64_t>(blockIdx.x) + 1) * split / gridDim.x;
  if (tb >= te && !pooled) return;
  // static part of the range; the rest went to the tail pool
  const int64_t ts = a.pool ? tb + (te - tb) * a.static_q / 1024 : te;
  const uint32_t smem0 = smem_addr(smem);

  // ------------------------------------------------------------ producer --
  // One thread (lane 0 of the last warp) fills the ring.  Its state:
  uint64_t pol = 0;  // L2 policy of the bulk copies
  int pk = -1;       // tensor of tile t
  TensorDesc d{};
  const void* gp = nullptr;
  TensorAux ax{nullptr, nullptr, 1.0f, 0};
  int32_t e_cur = 0;
  uint32_t amax_now = 0u, seed = 0u;
  int rot = 0;
  int64_t tiles = 0;
  int64_t t = tb, t_end = ts;  // the current run of consecutive tiles
  int ps = 0;                  // next stage to fill, and how many times the ring has wrapped
  uint32_t puse = 0;
  int64_t issued = 0;
  auto load = [&](int kk) {
    pk = kk;
    d = desc_of(a, pk);
    gp = grad_of(a, pk);
    if (WD != kBF16 && a.aux) ax = aux_of(a, pk);  // the launch has aux entries (inline ones too, when it carries its tables)
    tiles = (d.numel + kTile - 1) / kTile;
    if (WD == kE4M3) {
      const int64_t n = a.n_tensors;
      e_cur = a.fp8_exp[a.e_cur_slot * n + d.ring];
      amax_now = a.fp8_amax[a.a_cur_slot * n + d.ring];
      // The tensor's maximum flushed so far in this step, read through L2:
      // the slot was zeroed before this step and is raised only with exact
      // values, so it seeds the recomputation threshold after a tensor change
      // (under the tail pool a CTA changes tensor at almost every chunk).
      asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(seed) : "l"(a.fp8_amax + a.a_next_slot * n + d.ring) : "memory");
    }
    if (a.n_inline == 0 && d.tile_off + tiles < a.tile_base + T) {  // the next tensor's entries, into L1
      asm volatile("prefetch.global.L1 [%0];" ::"l"(a.desc + pk + 1));
      asm volatile("prefetch.global.L1 [%0];" ::"l"(a.grads + pk + 1));
      if (WD != kBF16 && a.aux) asm volatile("prefetch.global.L1 [%0];" ::"l"(a.aux + pk + 1));
    }
  };
  auto issue = [&]() {  // the copies of tile t (of tensor pk) into stage ps, which is free
    const int64_t e0 = (t - d.tile_off) * kTile;
    const int count = static_cast<int>(d.numel - e0 < kTile ? d.numel - e0 : kTile);
    // NVFP4 weights: half a byte per element (tile starts stay 16-byte aligned: 1920 bytes per tile)
    // what is copied of the weights and gradients: lo | hi << 16, from the region's start
    const uint32_t wr = WD == kNVFP4 ? staged_bytes(d.w, (count + 1) / 2, 1) << 16
                        : MIS && WD != kBF16 ? staged_range(d.w, d.numel, e0, count, WS)
                                             : staged_bytes(d.w, count, WS) << 16;
    const uint32_t gr = MIS ? staged_range(gp, d.numel, e0, count, GS) : staged_bytes(gp, count, GS) << 16;
    const uint32_t nw = (wr >> 16) - (MIS ? wr & 0xFFFFu : 0u), ng = (gr >> 16) - (MIS ? gr & 0xFFFFu : 0u);
    const uint32_t nm = staged_bytes(d.m, count, MS), nv = staged_bytes(d.v, count, MS);
    const uint32_t nve = staged_bytes(d.ve, count, MS);
    const int64_t s0 = WD == kE4M3B ? 2 * (e0 / kBlock) : e0 / kFp4Block;  // the tile's first scale byte
    const uint8_t* sp = static_cast<const uint8_t*>(ax.scale);
    const uint32_t ns = WD == kE4M3B   ? staged_bytes(sp + s0, 2 * ((count + kBlock - 1) / kBlock), 1)
                        : WD == kNVFP4 ? staged_bytes(sp + s0, (count + kFp4Block - 1) / kFp4Block, 1)
                                       : 0u;
    const uint32_t bar = smem_addr(&full_bar[ps]);
    const uint32_t st = smem0 + static_cast<uint32_t>(ps * a.stage_bytes);
    mbar_expect_tx(bar, nw + ng + nm + nv + nve + ns);
    const uint32_t wlo = MIS ? wr & 0xFFFFu : 0u, glo = MIS ? gr & 0xFFFFu : 0u;
    if (nw)
      tma_load(st + wlo, static_cast<const uint8_t*>(d.w) + (WD == kNVFP4 ? e0 / 2 : e0 * WS) -
                             (MIS && WD != kBF16 ? misalign(d.w) : 0u) + wlo, nw, bar, pol);
    if (ng)
      tma_load(st + a.off_g + glo, static_cast<const uint8_t*>(gp) + e0 * GS - (MIS ? misalign(gp) : 0u) + glo, ng,
               bar, pol);
    if (nm) tma_load(st + a.off_m, static_cast<const uint8_t*>(d.m) + e0 * MS, nm, bar, pol);
    if (nv) tma_load(st + a.off_v, static_cast<const uint8_t*>(d.v) + e0 * MS, nv, bar, pol);
    if (nve) tma_load(st + a.off_ve, static_cast<const uint8_t*>(d.ve) + e0 * MS, nve, bar, pol);
    if (ns) tma_load(st + a.off_s, sp + s0, ns, bar, pol);
    StageHead& hd = heads[ps];
    hd.w = d.w; hd.m = d.m; hd.v = d.v; hd.ve = d.ve;
    hd.g = gp;
    if (WD != kBF16) { hd.scale = ax.scale; hd.cc = ax.compute; hd.gscale = ax.gscale; }
    hd.goff = d.goff;
    hd.e0 = e0;
    hd.k = pk;
    hd.count = count;
    hd.rot = rot;
    hd.ring = d.ring;
    if (WD == kE4M3) { hd.e_cur = e_cur; hd.amax = amax_now; hd.seed = seed; }
    if (MIS) { hd.w_range = wr; hd.g_range = gr; }
    mbar_arrive(bar);  // publishes the head (release); the copies complete the phase
    // the next tile's first 256 elements go to the warp after this tile's
    // last: short tensors spread over the warps instead of all taking the first
    rot += (count + 32 * kGroup - 1) / (32 * kGroup);
    if (rot >= kConsumerWarps) rot -= kConsumerWarps;
    ++issued;
    ++t;
    if (++ps == S) { ps = 0; ++puse; }
  };
  if (tid == kConsumers) {
    // The producer sets up the ring and issues the copies of its first tile
    // before the block-wide barrier, in straight-line code next to the
    // kernel's entry: on a launch of a tile or two per CTA these copies are
    // on the critical path (issued 1.3 us after entry, against 2.0 us from
    // the loop below after the barrier).
    for (int i = 0; i < S; ++i) {
      mbar_init(smem_addr(&full_bar[i]), 1);
      mbar_init(smem_addr(&empty_bar[i]), kConsumerWarps);
    }
    mbar_init_fence();
    pol = evict_first_policy();
  }
  // Nothing of global memory is touched before the work ahead in the stream is
  // complete: the previous step, the kernels that wrote the gradients or the
  // tables.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (tid == kConsumers) {
    if (t < t_end) {
      load(first_tensor(a, tb));
      while (t >= d.tile_off + tiles) load(pk + 1);
      issue();
    }
  }
  __syncthreads();

  if (warp == kConsumerWarps) {
    if (lane != 0) return;
    // Every CTA's claims end with one beyond the pool, pool_chunks + gridDim.x
    // in all: the last of them wraps the counter back to 0 (a memset before
    // every launch cost a gap of its own on the stream).  A CTA that gives up
    // makes fewer: reading the launch's status clears the counters.
    auto claim = [&]() { return atomicInc(a.pool_next, static_cast<uint32_t>(a.pool_chunks) + gridDim.x - 1u); };
    bool failed = false;
    bool ahead = false;  // a claim (j) made before the run in hand is done
    uint32_t j = 0u;
    for (;;) {
      if (t >= t_end) {  // static part done: next chunk of the tail pool, if any
        if (!pooled) break;
        if (!ahead) j = claim();
        ahead = false;
        if (j >= static_cast<uint32_t>(a.pool_chunks)) break;
        int first;
        if (a.pool) {
          const PoolChunk pc = a.pool[j];
          t = pc.start;
          t_end = pc.start + pc.count;
          first = pc.first;
        } else {  // a pool without a table: the last tiles of the list, pool_len at a time
          t = a.pool_base + static_cast<int64_t>(j) * a.pool_len;
          t_end = t + a.pool_len < a.tile_base + T ? t + a.pool_len : a.tile_base + T;
          first = tensor_of(a, pk < 0 ? 0 : pk, t);
        }
        if (first != pk) load(first);
      }
      while (t >= d.tile_off + tiles) load(pk + 1);
      if (pooled && !ahead && t + 1 >= t_end) {  // the run's last tile: its wait for a free stage covers the claim's
        j = claim();
        ahead = true;
      }
      if (puse > 0 && !mbar_wait(smem_addr(&empty_bar[ps]), (puse - 1) & 1u)) {
        if (a.err) atomicOr(a.err, kErrEmptyWait);
        failed = true;
        break;
      }
      issue();
    }
    if (failed) {  // wait (bounded) for this CTA's copies still in flight, then leave
      const int64_t last = issued < S ? issued : S;
      for (int64_t i = 1; i <= last; ++i) {
        const int64_t it = issued - i;
        if (!mbar_wait(smem_addr(&full_bar[it % S]), static_cast<uint32_t>((it / S) & 1)) && a.err)
          atomicOr(a.err, kErrDrainWait);
      }
      return;
    }
    // no more work: once the next stage is free, post the end marker there
    if (puse > 0 && !mbar_wait(smem_addr(&empty_bar[ps]), (puse - 1) & 1u)) {
      if (a.err) atomicOr(a.err, kErrEmptyWait);
      return;
    }
    heads[ps].k = -1;
    mbar_arrive(smem_addr(&full_bar[ps]));
    if (pooled && blockIdx.x == 0) *a.pool_clear = 0u;
    return;
  }

  // ----------------------------------------------------------- consumers --
  const int n = a.n_tensors;
  int k = -1;
  TensorCtx x;
  int32_t e_next = 0;
  auto enter = [&](const StageHead& hd) {  // take up the stage's tensor
    k = hd.k;
    load_tensor<WD, GD, MD, MIS>(hd, x);
    if (WD == kE4M3) {
      e_next = fp8_next_exponent(hd.amax, hd.e_cur);
      x.dec_scale = pow2f(hd.e_cur);
      x.enc_scale = pow2f(-e_next);
      x.cc_scale = pow2f(e_next);
      x.amax_seed = __uint_as_float(hd.seed);
    }
  };
  uint32_t amax_bits = 0u;
  int s = 0;
  uint32_t use = 0;
  for (;;) {
    if (!__all_sync(0xFFFFFFFFu, mbar_wait(smem_addr(&full_bar[s]), use & 1u))) {  // warp-uniform give-up
      if (a.err && lane == 0) atomicOr(a.err, kErrFullWait);
      return;
    }
    const StageHead& hd = heads[s];
    const int kt = hd.k;
    if (kt < 0) break;  // the producer's end marker
    const int count = hd.count;
    const int lw = warp - hd.rot + (warp < hd.rot ? kConsumerWarps : 0);  // this warp's place in the tile
    const int c = 32 * lw + lane;  // consumer: elements [8c, 8c + 8) of the tile
    if (32 * kGroup * lw >= count) {  // nothing for this warp
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_addr(&empty_bar[s]));
      if (++s == S) { s = 0; ++use; }
      continue;
    }
    if (kt != k) {  // another tensor: flush this one's E4M3 amax
      if (WD == kE4M3 && k >= 0) {
        if (lane == 0 && amax_bits != 0u)
          atomicMax(&a.fp8_amax[static_cast<int64_t>(a.a_next_slot) * n + x.d.ring], amax_bits);
        amax_bits = 0u;
      }
      enter(hd);
    }
    const int64_t tile_e0 = hd.e0;
    if (WD == kE4M3 && tile_e0 == 0 && c == 0) {  // the CTA holding the tensor's first tile
      a.fp8_exp[static_cast<int64_t>(a.e_next_slot) * n + x.d.ring] = e_next;
      a.fp8_amax[static_cast<int64_t>(a.a_zero_slot) * n + x.d.ring] = 0u;
    }
    // Straight-line group: every array aligned, and this warp's 256 elements
    // all inside the tile (every warp of a whole tile; the whole warps of a
    // tensor's last tile, whose bytes the producer staged as well).  A warp
    // that holds the end of a partial tile takes the element-wise path below.
    if (x.fast && kGroup * 32 * (lw + 1) <= count) {
      const uint32_t st = smem0 + static_cast<uint32_t>(s * a.stage_bytes);
      const int64_t e0 = tile_e0 + kGroup * c;
      float w[8], g[8], m[8], v[8], ve[8];
      uint32_t h_old = 0u;
      if (MIS && (x.gsh | x.wsh) != 0u) patch_group<WD, GD>(a, x, hd, e0, c, st);
      if (WD == kBF16) {
        get_bf16(w, st + kGroup * WS * c);
      } else if (WD == kE4M3) {
        get_e4m3(w, st + x.wsh + kGroup * WS * c, x.dec_scale);
      } else if (WD == kE4M3B) {
        h_old = lds_u16(st + a.off_s + 2 * (c >> 2));
        get_e4m3(w, st + x.wsh + kGroup * WS * c, fp16_value(h_old));
      } else {
        h_old = lds_u8(st + a.off_s + (c >> 1));
        get_fp4(w, st + 4 * c, __fmul_rn(e4m3_value(h_old), x.gscale));
      }
      if (MIS && x.gsh != 0u) {
        if (GD == kF32) get_f32_at(g, st + a.off_g + x.gsh + kGroup * GS * c);
        else get_bf16_at(g, st + a.off_g + x.gsh + kGroup * GS * c);
      } else {
        if (GD == kF32) get_f32(g, st + a.off_g + kGroup * GS * c);
        else get_bf16(g, st + a.off_g + kGroup * GS * c);
      }
      if (MD == kF32) {
        get_f32(m, st + a.off_m + kGroup * MS * c);
        get_f32(v, st + a.off_v + kGroup * MS * c);
        get_f32(ve, st + a.off_ve + kGroup * MS * c);
      } else {
        get_bf16(m, st + a.off_m + kGroup * MS * c);
        get_bf16(v, st + a.off_v + kGroup * MS * c);
        get_bf16(ve, st + a.off_ve + kGroup * MS * c);
      }
      if constexpr (WD == kNVFP4 && MD == kF32) {
        // released at once: the rare exact branch re-reads global memory
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_addr(&empty_bar[s]));
        finish_fp4<GD, MD, SR, OPT, kExactGlobal>(a, x, e0, kGroup, h_old, w, g, m, v, ve, st, c);
      } else if constexpr (WD == kNVFP4) {
        // BF16 moments: the stage stays until the group is done (its exact
        // branch re-reads the binary32 originals there)
        finish_fp4<GD, MD, SR, OPT, kExactStage>(a, x, e0, kGroup, h_old, w, g, m, v, ve, st, c);
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_addr(&empty_bar[s]));
      } else {
        // the stage stays until the group is done: the rare exact branch reads
        // its inputs there
        if constexpr (WD == kE4M3B) finish_block<GD, MD, SR, OPT, true>(a, x, e0, kGroup, h_old, w, g, m, v, ve, st, c);
        else finish_group<WD, GD, MD, SR, OPT, true>(a, x, e0, kGroup, w, g, m, v, ve, amax_bits, st, c);
        __syncwarp();
        // one running maximum per warp: the lanes' own would each reach the
        // threshold again and again, in nearly every tile of some lane
        if (WD == kE4M3) amax_bits = __reduce_max_sync(0xFFFFFFFFu, amax_bits);
        if (lane == 0) mbar_arrive(smem_addr(&empty_bar[s]));
      }
      if (++s == S) { s = 0; ++use; }
      continue;
    }
    // partial tile or unstaged arrays: element-wise fallback (inline or a
    // call, by moment format; the NVFP4 one is always a call: inline it slowed
    // the stochastic-rounding loop by 5 %)
    if constexpr (WD == kE4M3B) {
      if constexpr (MD == kF32)
        general_block_group<GD, MD, SR, OPT, MIS>(a, x, hd, tile_e0, count, c, smem0 + static_cast<uint32_t>(s * a.stage_bytes));
      else
        general_block_group_call<GD, MD, SR, OPT, MIS>(a, x, hd, tile_e0, count, c,
                                                  smem0 + static_cast<uint32_t>(s * a.stage_bytes));
    } else if constexpr (WD == kNVFP4)
      general_fp4_group<GD, MD, SR, OPT>(a, x, hd, tile_e0, count, c, smem0 + static_cast<uint32_t>(s * a.stage_bytes));
    else
      amax_bits = MD == kF32 ? general_group<WD, GD, MD, SR, OPT, MIS>(a, x, hd, tile_e0, count, c,
                                                                   smem0 + static_cast<uint32_t>(s * a.stage_bytes),
                                                                   amax_bits)
                             : general_group_call<WD, GD, MD, SR, OPT, MIS>(
                                   a, x, hd, tile_e0, count, c, smem0 + static_cast<uint32_t>(s * a.stage_bytes), amax_bits);
    __syncwarp();
    if (WD == kE4M3) amax_bits = __reduce_max_sync(0xFFFFFFFFu, amax_bits);
    if (lane == 0) mbar_arrive(smem_addr(&empty_bar[s]));
    if (++s == S) { s = 0; ++use; }
  }
  if (WD == kE4M3 && k >= 0 && lane == 0 && amax_bits != 0u)
    atomicMax(&a.fp8_amax[static_cast<int64_t>(a.a_next_slot) * n + x.d.ring], amax_bits);
}

}  // namespace mpadam
