// Shared device helpers for the sm_103a kernels: bf16 packing, mbarrier, TMA and
// tcgen05 (5th-generation tensor core, TMEM) wrappers written as inline PTX from the
// public PTX ISA.  Every spin-wait here is bounded: it gives up after
// kWaitTimeoutNs of %globaltimer time, raises a CTA-local abort flag and records a
// code in the device status word so the host can report SGD_ERR_DEVICE_TIMEOUT.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace sgd {

using bf16 = __nv_bfloat16;
using f16 = __half;

constexpr uint64_t kWaitTimeoutNs = 2000000000ull;  // 2 s: far above any legitimate wait

// ----------------------------------------------------------------------------
// bf16 helpers
// ----------------------------------------------------------------------------

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void unpack_bf16x8(const uint4& u, float* f) {
  const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float2 t = __bfloat1622float2(p[i]);
    f[2 * i] = t.x;
    f[2 * i + 1] = t.y;
  }
}

__device__ __forceinline__ uint4 pack_bf16x8(const float* f) {
  uint4 u;
  u.x = pack_bf16x2(f[0], f[1]);
  u.y = pack_bf16x2(f[2], f[3]);
  u.z = pack_bf16x2(f[4], f[5]);
  u.w = pack_bf16x2(f[6], f[7]);
  return u;
}

// Raised when an fp16 store had to clamp a value (|x| > 65504, or NaN) — one instance per
// translation unit (internal linkage), read and cleared by the host through
// f16_clamp_flag_here() of that unit.
static __device__ unsigned int g_f16_clamped;

// fp16 operands: values are clamped to the finite fp16 range before rounding so that
// an out-of-range activation saturates instead of turning into inf / NaN downstream; the
// clamp raises g_f16_clamped, which sgd_check_device reports.
__device__ __forceinline__ float sat_f16(float x) {
  if (!(fabsf(x) <= 65504.f)) g_f16_clamped = 1u;
  return fminf(fmaxf(x, -65504.f), 65504.f);
}

__device__ __forceinline__ uint32_t pack_f16x2(float lo, float hi) {
  __half2 v = __floats2half2_rn(sat_f16(lo), sat_f16(hi));
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void unpack_f16x8(const uint4& u, float* f) {
  const __half2* p = reinterpret_cast<const __half2*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float2 t = __half22float2(p[i]);
    f[2 * i] = t.x;
    f[2 * i + 1] = t.y;
  }
}

// max(|a|, |b|, |c|), NaN if any is NaN (one instruction on sm_100 and later)
__device__ __forceinline__ float absmax3_nan(float a, float b, float c) {
  float d;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Eight values as pack_f16x2 rounds and clamps them.  The clamp is rare, so the eight are
// checked together (four instructions instead of four per value) and rounded as they are
// unless one of them is out of range: packing was most of the instructions of an fp16
// epilogue.
__device__ __forceinline__ uint4 pack_f16x8(const float* f) {
  const float m = absmax3_nan(absmax3_nan(f[0], f[1], f[2]), absmax3_nan(f[3], f[4], f[5]), absmax3_nan(f[6], f[7], 0.f));
  uint4 u;
  if (m <= 65504.f) {
    const __half2 h0 = __floats2half2_rn(f[0], f[1]), h1 = __floats2half2_rn(f[2], f[3]);
    const __half2 h2 = __floats2half2_rn(f[4], f[5]), h3 = __floats2half2_rn(f[6], f[7]);
    u.x = *reinterpret_cast<const uint32_t*>(&h0);
    u.y = *reinterpret_cast<const uint32_t*>(&h1);
    u.z = *reinterpret_cast<const uint32_t*>(&h2);
    u.w = *reinterpret_cast<const uint32_t*>(&h3);
    return u;
  }
  u.x = pack_f16x2(f[0], f[1]);
  u.y = pack_f16x2(f[2], f[3]);
  u.z = pack_f16x2(f[4], f[5]);
  u.w = pack_f16x2(f[6], f[7]);
  return u;
}

__device__ __forceinline__ uint2 pack_f16x4(float4 f) {
  const float m = absmax3_nan(absmax3_nan(f.x, f.y, f.z), f.w, 0.f);
  uint2 u;
  if (m <= 65504.f) {
    const __half2 h0 = __floats2half2_rn(f.x, f.y), h1 = __floats2half2_rn(f.z, f.w);
    u.x = *reinterpret_cast<const uint32_t*>(&h0);
    u.y = *reinterpret_cast<const uint32_t*>(&h1);
    return u;
  }
  u.x = pack_f16x2(f.x, f.y);
  u.y = pack_f16x2(f.z, f.w);
  return u;
}

// SiLU and tanh-GELU as x * sigmoid(.) with the fast exponential and division intrinsics:
// 0.5 x (1 + tanh(u)) = x / (1 + e^(-2u)), which has no cancellation for negative x (the
// libm tanhf / expf calls made the activation the longest part of the epilogue of a
// short-K MLP projection).  An overflowing e^(.) gives x / inf = 0, the limit.
__device__ __forceinline__ float silu_f(float x) { return __fdividef(x, 1.0f + __expf(-x)); }
__device__ __forceinline__ float gelu_erf_f(float x) {
  return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_tanh_f(float x) {
  const float c2 = 2.0f * 0.79788456080286536f;  // 2 sqrt(2/pi)
  return __fdividef(x, 1.0f + __expf(-c2 * (x + 0.044715f * x * x * x)));
}

// Pairs of fp32 values in 64 bits: one instruction for two rounded-to-nearest fp32 results.
__device__ __forceinline__ uint64_t pack_f32x2(uint32_t lo, uint32_t hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
  return d;
}
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
  return pack_f32x2(__float_as_uint(lo), __float_as_uint(hi));
}
__device__ __forceinline__ float lo_f32x2(uint64_t a) { return __uint_as_float(static_cast<uint32_t>(a)); }
__device__ __forceinline__ float hi_f32x2(uint64_t a) { return __uint_as_float(static_cast<uint32_t>(a >> 32)); }
__device__ __forceinline__ float sum_f32x2(uint64_t a) { return lo_f32x2(a) + hi_f32x2(a); }
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// max of three (a NaN is ignored, as by fmaxf)
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// 2^x with the hardware's approximate base-2 exponential (PTX ex2.approx.ftz.f32).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// x0 / (1 + 2^t0) and x1 / (1 + 2^t1) with one reciprocal, r = 1 / (d0 d1): the special-function unit
// (an exponential and a reciprocal per value) bounded the GELU and SwiGLU epilogues.  Above
// t = 62 the factor is taken as 0 (it is under 2^-62; x times it is x / inf in the limit, NaN for an
// infinite x), and the exponents are held there so that d0 d1 stays in range.
__device__ __forceinline__ void sigmoid_scale2(float& x0, float& x1, float t0, float t1) {
  const float d0 = 1.0f + ex2_approx(fminf(t0, 62.f)), d1 = 1.0f + ex2_approx(fminf(t1, 62.f));
  const float r = __fdividef(1.0f, d0 * d1);
  x0 *= t0 > 62.f ? 0.f : r * d1;
  x1 *= t1 > 62.f ? 0.f : r * d0;
}
__device__ __forceinline__ void silu2(float& x0, float& x1) {
  constexpr float k = -1.4426950408889634f;  // -log2(e)
  sigmoid_scale2(x0, x1, k * x0, k * x1);
}
__device__ __forceinline__ void gelu_tanh2(float& x0, float& x1) {
  constexpr float k0 = -2.0f * 0.79788456080286536f * 1.4426950408889634f;  // -2 sqrt(2/pi) log2(e)
  constexpr float k1 = 0.044715f * k0;
  sigmoid_scale2(x0, x1, x0 * fmaf(k1, x0 * x0, k0), x1 * fmaf(k1, x1 * x1, k0));
}

// ----------------------------------------------------------------------------
// shared-memory addresses, timers
// ----------------------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t lane_id() {
  uint32_t l;
  asm volatile("mov.u32 %0, %%laneid;" : "=r"(l));
  return l;
}

// ----------------------------------------------------------------------------
// programmatic dependent launch (PTX griddepcontrol)
// ----------------------------------------------------------------------------

// Wait until the grids this grid depends on have completed and their memory is visible
// (returns at once for a grid launched without programmatic serialization), then let the
// next grid in the stream begin launching (its CTAs run their own prologue and wait here in
// turn).  Every kernel of a step program calls this after its shared-memory / TMEM-only
// prologue and before its first global-memory access (but for the group GEMM's first loads of
// its weight, which no kernel of a step program writes).
__device__ __forceinline__ void pdl_wait_and_trigger() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Four floats of what an earlier kernel of the step wrote (16-byte aligned).  A kernel of a step is
// resident while its predecessor still writes, so that such data is not read-only for the kernel's
// lifetime, as __ldg (ld.global.nc) demands: __ldg is for weights and tables alone.  As an
// asm volatile the load stays behind pdl_wait_and_trigger but may pass stores to shared memory.
__device__ __forceinline__ float4 ld_f32x4(const float* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(__cvta_generic_to_global(p)));
  return v;
}

// ----------------------------------------------------------------------------
// mbarrier
// ----------------------------------------------------------------------------

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// A wait looks at the abort flag and at %globaltimer (whose read stalls the reading thread for
// hundreds of clocks) once in kPollsPerTimer polls, so that a wait of the usual length only polls.
constexpr uint32_t kPollsPerTimer = 256;

__device__ __forceinline__ bool wait_expired(uint64_t& t0) {
  const uint64_t now = global_timer_ns();
  if (t0 == 0) t0 = now;
  return now - t0 > kWaitTimeoutNs;
}

// Wait for the phase with parity `parity` of `bar` to complete.  Returns false (and
// leaves the barrier alone) if the CTA-wide abort flag is raised or the wait exceeds
// kWaitTimeoutNs; in the latter case it raises the flag and records `code` in
// *status.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          int* status, int code) {
  uint64_t t0 = 0;
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if (i % kPollsPerTimer == 0) {
      if (*abort_flag) return false;
      if (wait_expired(t0)) {
        *abort_flag = 1;
        if (status) atomicCAS(status, 0, code);
        return false;
      }
    }
  }
}

// The same wait by a whole converged warp, on a shared-memory address; returns the same value
// in every lane (so that the compiler keeps what follows warp-uniform).
__device__ __forceinline__ bool mbar_try_wait_at(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               int* status, int code) {
  uint64_t t0 = 0;
  for (uint32_t i = 1;; ++i) {
    if (__all_sync(0xffffffffu, mbar_try_wait_at(bar, parity))) return true;
    if (i % kPollsPerTimer == 0) {
      int stop = *abort_flag;
      if (!stop && wait_expired(t0)) {
        *abort_flag = stop = 1;
        if (status) atomicCAS(status, 0, code);
      }
      if (__any_sync(0xffffffffu, stop)) return false;
    }
  }
}

// Bounded wait that ignores the abort flag (used while draining after an abort).
__device__ __forceinline__ void mbar_drain(uint64_t* bar, uint32_t parity) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > kWaitTimeoutNs) break;
  }
}

// Whether the phase with parity `parity` has completed, without waiting (all lanes alike).
__device__ __forceinline__ bool mbar_test_warp(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return __all_sync(0xffffffffu, ok != 0);
}

// One lane of a converged warp, the same on every call.
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok));
  return ok != 0;
}

__device__ __forceinline__ void mbar_arrive_expect_tx_at(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// ----------------------------------------------------------------------------
// TMA (cp.async.bulk.tensor)
// ----------------------------------------------------------------------------

__device__ __forceinline__ void tma_prefetch_desc(const void* desc) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(desc)) : "memory");
}

// 2-D tiled load of the box at (c0 = inner/column, c1 = row) into shared memory; the
// transaction bytes are credited to `bar`.
__device__ __forceinline__ void tma_load_2d(void* smem_dst, const void* desc, uint64_t* bar, int c0,
                                            int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(desc)), "r"(smem_u32(bar)), "r"(c0), "r"(c1)
      : "memory");
}

// The same with shared-memory addresses.
__device__ __forceinline__ void tma_load_2d_at(uint32_t dst, const void* desc, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(desc)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}

// Plain bulk copy of `bytes` (a multiple of 16; both addresses 16-byte aligned) into shared memory.
__device__ __forceinline__ void bulk_load(void* smem_dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(smem_dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// ----------------------------------------------------------------------------
// tcgen05: TMEM allocation, MMA, commit, loads
// ----------------------------------------------------------------------------

__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
}

__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// D[tmem] (+)= A[smem] * B[smem]^T, f16 x f16 -> fp32, shape from idesc.
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                          uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Same with A read from Tensor Memory (M rows in TMEM lanes, two fp16 K-elements per
// 32-bit column, the lower K index in the low half): 8 columns per K = 16 slice.
__device__ __forceinline__ void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                             uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrive once on `bar` when every tcgen05.mma issued so far by this thread completes.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void umma_commit_at(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}

// 32 lanes x 32 bits, 16 consecutive columns per thread.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

// Wait for this thread's outstanding tcgen05.ld; the register operands tie the
// consumers of the loaded values to after the wait.
__device__ __forceinline__ void tmem_ld_wait16(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                 "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                 "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

// Store 16 consecutive columns of this thread's TMEM lane (32 lanes x 32 bits).
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

__device__ __forceinline__ void tmem_st_wait() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Make this thread's generic-proxy shared-memory writes visible to the async proxy
// (tensor-core operand reads) before signalling the MMA issuer.
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Shared-memory matrix descriptor for a K-major operand tile written by TMA with
// 128-byte swizzling: rows of 128 B, 8-row groups 1024 B apart (stride byte offset),
// descriptor version 1, layout SWIZZLE_128B.  The leading byte offset is not used by
// swizzled K-major layouts.  The tile base must be 1024-byte aligned; the K slice k
// of a 64-element row block starts 32 k bytes further.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);  // start address, bits [0,14)
  d |= static_cast<uint64_t>(1) << 16;                   // leading byte offset (unused)
  d |= static_cast<uint64_t>(1024 >> 4) << 32;           // stride byte offset, bits [32,46)
  d |= static_cast<uint64_t>(1) << 46;                   // descriptor version
  d |= static_cast<uint64_t>(2) << 61;                   // SWIZZLE_128B
  return d;
}

// Same for 64-byte rows written with 64-byte swizzling (8-row groups 512 B apart,
// layout SWIZZLE_64B); the K slice k of a 32-element row starts 32 k bytes further.
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t saddr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;
  d |= static_cast<uint64_t>(512 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(4) << 61;                   // SWIZZLE_64B
  return d;
}

// Same for 32-byte rows written with 32-byte swizzling (8-row groups 256 B apart, layout
// SWIZZLE_32B): one K = 16 slice per 32-byte row.
__device__ __forceinline__ uint64_t smem_desc_sw32(uint32_t saddr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;
  d |= static_cast<uint64_t>(256 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(6) << 61;                   // SWIZZLE_32B
  return d;
}

// MN-major operand in 32-byte swizzle atoms of 8 K-rows x 16 fp16: `lbo` = bytes between
// atoms along N, `sbo` = bytes between 8-row groups along K.
__device__ __forceinline__ uint64_t smem_desc_sw32_mn(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(6) << 61;
  return d;
}

// Shared-memory descriptor for an MN-major operand (the N index contiguous) stored as
// 128-byte swizzle atoms of 8 K-rows x 64 fp16: `lbo` = bytes between atoms along N,
// `sbo` = bytes between 8-row groups along K.
__device__ __forceinline__ uint64_t smem_desc_sw128_mn(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}

// Instruction descriptor of tcgen05.mma kind::f16: fp32 accumulator, fp16 A and B
// (format code 0 in both fields; A and B always share one type), both K-major, M x N.
__host__ __device__ constexpr uint32_t umma_idesc_f16(int M, int N) {
  return (1u << 4)                                   // D format: f32
         | (0u << 7)                                 // A format: f16
         | (0u << 10)                                // B format: f16
         | (static_cast<uint32_t>(N >> 3) << 17)     // N / 8
         | (static_cast<uint32_t>(M >> 4) << 24);    // M / 16
}

// Same with B MN-major (transpose-B bit 16): B stored with its N index contiguous.
__host__ __device__ constexpr uint32_t umma_idesc_f16_bmn(int M, int N) {
  return umma_idesc_f16(M, N) | (1u << 16);
}

// ----------------------------------------------------------------------------
// CTA pairs (clusters of two; tcgen05 cta_group::2)
// ----------------------------------------------------------------------------

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// shared::cluster address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}

// Barrier over every thread of the cluster (all of them reach it: every other wait is bounded).
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// tma_load_2d_at into this CTA's shared memory whose bytes are credited to a barrier of either
// CTA of the pair (a shared::cluster address).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const void* desc, uint32_t cluster_bar, int c0,
                                                 int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(desc)), "r"(cluster_bar), "r"(c0), "r"(c1)
      : "memory");
}

// Both CTAs of the pair allocate (and free) together, one warp each.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// D (256 rows: 128 in each CTA's TMEM) (+)= A B^T: each CTA's shared memory holds its 128 rows of
// A and its half of B's rows at the descriptors' addresses.  Issued by the leader (rank 0).
__device__ __forceinline__ void umma_f16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                              uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrive once on the barrier at this shared-memory offset in both CTAs when every MMA issued so
// far by this thread has completed.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          bar),
      "h"(static_cast<uint16_t>(3))
      : "memory");
}

// Every translation unit registers its clamp flag's accessor at load time; the host reads
// them all (sgd_kernel_f16_clamped).  Defined in api.cu.
int register_f16_clamp_flag(unsigned int* (*accessor)());

// Device address of this translation unit's clamp flag on the current device (cached per
// device; nullptr if it cannot be obtained).
static inline unsigned int* f16_clamp_flag_here() {
  static unsigned int* ptr[64] = {nullptr};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  if (!ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_f16_clamped) != cudaSuccess) return nullptr;
    ptr[dev] = static_cast<unsigned int*>(p);
  }
  return ptr[dev];
}

static const int g_f16_clamp_registered = register_f16_clamp_flag(&f16_clamp_flag_here);

// Host: launches made while pdl_flag() is set (the kernels of a step program, see run_ops in
// api.cu) carry the programmatic-stream-serialization attribute, so that in a captured graph
// each kernel's launch and prologue overlap the tail of the one before (programmatic edges).
bool& pdl_flag();
int64_t& pdl_launches();  // the calling thread's launches with the attribute

template <typename... KArgs, typename... Args>
static inline cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                   cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  if (pdl_flag()) {
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    ++pdl_launches();
  }
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace sgd
