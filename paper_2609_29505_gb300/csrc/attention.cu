// Non-causal multi-head attention O = softmax(Q K^T / sqrt(d_h)) V, flash style.
//
// Used inside every active self-attention and cross-attention branch (Algorithm 2:
// an active unit evaluates F_l(h_{l-1,s}; c_s)); frozen units never launch it.
//
// Four kernels:
//   attn_pp_kernel (d_h 64, 72, 128; long or many sequences): tcgen05 with two query tiles per
//     CTA and two alternating softmax warpgroups, P in TMEM; described above the kernel.
//   attn_sm_kernel (d_h 64, 72, 128; few keys or an ill-fitting last wave, by attn_small): tcgen05
//     with one query tile per CTA, key tiles of 64, and several CTAs per SM.
//   attn_tc_kernel (d_h 64, 128): tcgen05.  One CTA = 128 queries of one (sample, head),
//     keys in tiles of 128.  Warp 0 loads Q once and K/V tiles through a 2-stage TMA ring;
//     warp 1 issues S = Q K^T into one of two TMEM S buffers and O += P V into a TMEM O
//     accumulator (V read as an MN-major operand straight from its row-major tile);
//     warps 2-5 (one query row per thread) read S from TMEM, run the online softmax in
//     fp32 and write P (fp16) into a 128-byte-swizzled shared tile for the next MMA.  O
//     is rescaled only when a row maximum grows by more than 2^8 (P <= 256 otherwise),
//     which keeps the result exact while avoiding most TMEM round trips.
//   attn_kernel (any of 64, 72, 128): mma.sync, described below; used for d_h = 72.
//
// mma.sync kernel: one CTA = 64 query rows of one (sample, head), 4 warps x 16 rows.  K/V tiles of
// 64 keys stream through a double-buffered cp.async ring; S = Q K^T and O += P V run
// on mma.sync m16n8k16 (fp16 in, fp32 accumulate) with an online softmax in
// registers (exp2 with the scale folded in).  Q, K, V, P and O are fp16 (m16n8k16
// f16 x f16 -> f32).  Keys beyond n_kv are masked and their
// shared-memory rows zero-filled; head dims 72 are padded to 80 in shared memory.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "common.cuh"
#include "kernels.h"

namespace sgd {

namespace {

constexpr int kBQ = 64;
constexpr int kBKV = 64;
constexpr int kWarps = 4;

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool valid) {
  const uint32_t s = smem_u32(smem);
  const int sz = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s), "l"(gmem), "r"(sz)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t* r, const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t* r, const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}

__device__ __forceinline__ void mma_f16_16816(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// DP: padded head dim in shared memory (multiple of 16); DH: real head dim.
template <int DH, int DP>
__global__ void __launch_bounds__(kWarps * 32) attn_kernel(const AttnParams p) {
  constexpr int kPitch = DP + 8;           // elements per shared row (bank-conflict free)
  constexpr int kChunks = DH / 8;          // 16-byte chunks of real data per row
  constexpr int kPadChunks = DP / 8;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  f16* sQ = reinterpret_cast<f16*>(smem_raw);
  f16* sK = sQ + kBQ * kPitch;            // [2][kBKV][kPitch]
  f16* sV = sK + 2 * kBKV * kPitch;       // [2][kBKV][kPitch]

  pdl_wait_and_trigger();
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int q0 = blockIdx.x * kBQ;
  const int bh = blockIdx.y;
  const int b = bh / p.n_heads, h = bh % p.n_heads;
  const int hs = p.head_stride > 0 ? p.head_stride : DH;  // input columns between heads
  const f16* qbase = p.q + (static_cast<int64_t>(b) * p.n_q) * p.ldq + h * hs;
  const f16* kbase = p.k + (static_cast<int64_t>(b) * p.n_kv) * p.ldkv + h * hs;
  const f16* vbase = p.v + (static_cast<int64_t>(b) * p.n_kv) * p.ldkv + h * hs;

  // Q tile
  for (int i = tid; i < kBQ * kPadChunks; i += kWarps * 32) {
    const int r = i / kPadChunks, c = i % kPadChunks;
    const bool ok = (q0 + r) < p.n_q && c < kChunks;
    const f16* src = ok ? qbase + static_cast<int64_t>(q0 + r) * p.ldq + c * 8 : p.q;
    cp_async16(sQ + r * kPitch + c * 8, src, ok);
  }
  auto load_kv = [&](int tile, int buf) {
    const int k0 = tile * kBKV;
    f16* dk = sK + buf * kBKV * kPitch;
    f16* dv = sV + buf * kBKV * kPitch;
    for (int i = tid; i < kBKV * kPadChunks; i += kWarps * 32) {
      const int r = i / kPadChunks, c = i % kPadChunks;
      const bool ok = (k0 + r) < p.n_kv && c < kChunks;
      const int64_t off = static_cast<int64_t>(k0 + r) * p.ldkv + c * 8;
      cp_async16(dk + r * kPitch + c * 8, ok ? kbase + off : p.k, ok);
      cp_async16(dv + r * kPitch + c * 8, ok ? vbase + off : p.v, ok);
    }
  };
  const int n_tiles = (p.n_kv + kBKV - 1) / kBKV;
  load_kv(0, 0);
  cp_async_commit();

  constexpr int KS = DP / 16;   // k-steps over the head dim
  constexpr int NO = DP / 8;    // output n-tiles
  uint32_t qf[KS][4];
  float o[NO][4];
#pragma unroll
  for (int i = 0; i < NO; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  float m_r[2] = {-INFINITY, -INFINITY}, l_r[2] = {0.f, 0.f};
  const float sl2 = 1.4426950408889634f / sqrtf(static_cast<float>(DH));  // log2(e)/sqrt(d_h)
  const int g = lane >> 2, t4 = lane & 3;

  for (int tile = 0; tile < n_tiles; ++tile) {
    const int buf = tile & 1;
    if (tile + 1 < n_tiles) {
      load_kv(tile + 1, buf ^ 1);
      cp_async_commit();
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    if (tile == 0) {
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const int r = warp * 16 + (lane & 15);
        const int c = ks * 16 + (lane >> 4) * 8;
        ldmatrix_x4(qf[ks], sQ + r * kPitch + c);
      }
    }
    const f16* tk = sK + buf * kBKV * kPitch;
    const f16* tv = sV + buf * kBKV * kPitch;
    // S = Q K^T : 16 x 64 per warp
    float s[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i][0] = s[i][1] = s[i][2] = s[i][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
#pragma unroll
      for (int np = 0; np < 4; ++np) {
        uint32_t kb[4];
        const int r = np * 16 + (lane & 7) + ((lane >> 4) << 3);
        const int c = ks * 16 + ((lane >> 3) & 1) * 8;
        ldmatrix_x4(kb, tk + r * kPitch + c);
        mma_f16_16816(s[2 * np], qf[ks], kb);
        mma_f16_16816(s[2 * np + 1], qf[ks], kb + 2);
      }
    }
    // mask keys beyond n_kv
    const int kbase_idx = tile * kBKV;
    if (kbase_idx + kBKV > p.n_kv) {
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        const int j = kbase_idx + nt * 8 + 2 * t4;
        if (j >= p.n_kv) { s[nt][0] = -INFINITY; s[nt][2] = -INFINITY; }
        if (j + 1 >= p.n_kv) { s[nt][1] = -INFINITY; s[nt][3] = -INFINITY; }
      }
    }
    // online softmax (rows g and g + 8 of this warp's 16)
    float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      mx[0] = fmaxf(mx[0], fmaxf(s[nt][0], s[nt][1]));
      mx[1] = fmaxf(mx[1], fmaxf(s[nt][2], s[nt][3]));
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
      mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
    }
    float corr[2], mnew[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      mnew[r] = fmaxf(m_r[r], mx[r]);
      corr[r] = exp2f((m_r[r] - mnew[r]) * sl2);
      m_r[r] = mnew[r];
    }
    float rs[2] = {0.f, 0.f};
    uint32_t pf[4][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const float p0 = exp2f((s[nt][0] - mnew[0]) * sl2);
      const float p1 = exp2f((s[nt][1] - mnew[0]) * sl2);
      const float p2 = exp2f((s[nt][2] - mnew[1]) * sl2);
      const float p3 = exp2f((s[nt][3] - mnew[1]) * sl2);
      rs[0] += p0 + p1;
      rs[1] += p2 + p3;
      const int kk = nt >> 1, hi = nt & 1;
      pf[kk][hi * 2 + 0] = pack_f16x2(p0, p1);
      pf[kk][hi * 2 + 1] = pack_f16x2(p2, p3);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      rs[r] += __shfl_xor_sync(0xffffffffu, rs[r], 1);
      rs[r] += __shfl_xor_sync(0xffffffffu, rs[r], 2);
      l_r[r] = l_r[r] * corr[r] + rs[r];
    }
#pragma unroll
    for (int i = 0; i < NO; ++i) {
      o[i][0] *= corr[0]; o[i][1] *= corr[0];
      o[i][2] *= corr[1]; o[i][3] *= corr[1];
    }
    // O += P V
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      // A fragment order: a0 (row g, k 0-7), a1 (row g+8, k 0-7), a2 (row g, k 8-15), a3
      uint32_t a[4] = {pf[kk][0], pf[kk][1], pf[kk][2], pf[kk][3]};
#pragma unroll
      for (int np = 0; np < NO / 2; ++np) {
        uint32_t vb[4];
        const int r = kk * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
        const int c = np * 16 + (lane >> 4) * 8;
        ldmatrix_x4_trans(vb, tv + r * kPitch + c);
        mma_f16_16816(o[2 * np], a, vb);
        mma_f16_16816(o[2 * np + 1], a, vb + 2);
      }
    }
    __syncthreads();
  }
  // normalise and store
  const float inv0 = 1.f / l_r[0], inv1 = 1.f / l_r[1];
  const int row0 = q0 + warp * 16 + g, row1 = row0 + 8;
  f16* ob = p.o + (static_cast<int64_t>(b) * p.n_q) * p.ldo + h * DH;
#pragma unroll
  for (int nt = 0; nt < NO; ++nt) {
    const int c = nt * 8 + 2 * t4;
    if (c < DH) {
      if (row0 < p.n_q)
        *reinterpret_cast<uint32_t*>(ob + static_cast<int64_t>(row0) * p.ldo + c) =
            pack_f16x2(o[nt][0] * inv0, o[nt][1] * inv0);
      if (row1 < p.n_q)
        *reinterpret_cast<uint32_t*>(ob + static_cast<int64_t>(row1) * p.ldo + c) =
            pack_f16x2(o[nt][2] * inv1, o[nt][3] * inv1);
    }
  }
}

// ----------------------------------------------------------------------------
// tcgen05 flash attention
// ----------------------------------------------------------------------------

constexpr int kTcThreads = 192;
constexpr int kTcBQ = 128;
constexpr int kTcBK = 128;
constexpr int kAtom = 128 * 64 * 2;  // 128 rows x 64 fp16: one 128-byte-swizzle column block
constexpr float kRescaleLog2 = 8.f;  // rescale O only when the row max grows by > 2^8

// fp16 pair, round to nearest, no saturation (the callers' values are far below 65504)
__device__ __forceinline__ uint32_t pack_f16x2_rn(float lo, float hi) {
  __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// The softmax of a query row in registers, where a thread's own instructions are the longest
// part of the chain S -> P -> O: three-input maxima and paired multiplications and additions.
template <int N>
__device__ __forceinline__ float row_max(const uint32_t* r) {
  float mx[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) mx[i] = fmaxf(__uint_as_float(r[i]), __uint_as_float(r[i + 8]));
#pragma unroll
  for (int c = 16; c < N; c += 16)
#pragma unroll
    for (int i = 0; i < 8; ++i) mx[i] = max3(mx[i], __uint_as_float(r[c + i]), __uint_as_float(r[c + 8 + i]));
  return fmaxf(max3(mx[0], mx[1], mx[2]), max3(max3(mx[3], mx[4], mx[5]), mx[6], mx[7]));
}

// P = 2^(score * scale - m2) of 32 scores, packed in place as fp16 pairs (pair k into register k, its
// scores already used), and their sums added to `sum` (four chains of pairs).
__device__ __forceinline__ void exp_pack32(uint32_t* r, uint64_t scale2, uint64_t neg_m2, uint64_t* sum) {
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const uint64_t t = fma_f32x2(pack_f32x2(r[2 * k], r[2 * k + 1]), scale2, neg_m2);
    const float p0 = ex2_approx(lo_f32x2(t)), p1 = ex2_approx(hi_f32x2(t));
    sum[k & 3] = add_f32x2(sum[k & 3], pack_f32x2(p0, p1));
    r[k] = pack_f16x2_rn(p0, p1);
  }
}

struct AttnTcArgs {
  CUtensorMap tmap_q;
  CUtensorMap tmap_k;
  CUtensorMap tmap_v;
  // d_h = 72 (heads padded to 80 columns in the input): boxes of the last 16 columns
  CUtensorMap tmap_q16;
  CUtensorMap tmap_k16;
  CUtensorMap tmap_v16;
  int head_stride;  // input columns between heads
  f16* o;
  int ldo;
  int n_q, n_kv, n_heads;
  float scale_log2;
  int* status;
};

template <int DH>
struct TcLayout {
  static constexpr int kAtoms = DH / 64;
  static constexpr int kQ = 0;
  static constexpr int kKV = kAtoms * kAtom;           // stage s: K atoms, then V atoms
  static constexpr int kStage = 2 * kAtoms * kAtom;
  static constexpr int kP = kKV + 2 * kStage;          // two P buffers of 128 keys
  static constexpr int kPBuf = 2 * kAtom;
  static constexpr int kBar = kP + 2 * kPBuf;
  static constexpr int kBytes = kBar + 256 + 1024;
  static constexpr uint32_t kTmemS = 0;                // S buffers at columns 0, 128
  static constexpr uint32_t kTmemO = 256;              // O at columns 256 .. 256 + DH
};

__device__ __forceinline__ bool warp_wait_bar(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                              int* status, int code) {
  int ok = 0;
  if (lane_id() == 0) ok = mbar_wait(bar, parity, abort_flag, status, code) ? 1 : 0;
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

template <int DH>
__global__ void __launch_bounds__(kTcThreads, 1) attn_tc_kernel(const __grid_constant__ AttnTcArgs a) {
  using L = TcLayout<DH>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + L::kBar);
  uint64_t* q_full = bars;
  uint64_t* kv_full = bars + 1;
  uint64_t* kv_empty = bars + 3;
  uint64_t* s_full = bars + 5;
  uint64_t* s_free = bars + 7;
  uint64_t* p_full = bars + 9;
  uint64_t* o_done = bars + 11;
  uint64_t* drain = bars + 13;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 14);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qt = blockIdx.x, bh = blockIdx.y;
  const int b = bh / a.n_heads, h = bh % a.n_heads;
  const int nt = (a.n_kv + kTcBK - 1) / kTcBK;

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&kv_full[i], 1);
      mbar_init(&kv_empty[i], 1);
      mbar_init(&s_full[i], 1);
      mbar_init(&s_free[i], 4);
      mbar_init(&p_full[i], 4);
      mbar_init(&o_done[i], 1);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&a.tmap_q);
    tma_prefetch_desc(&a.tmap_k);
    tma_prefetch_desc(&a.tmap_v);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait_and_trigger();  // the prologue above touched only shared memory and TMEM
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      mbar_arrive_expect_tx(q_full, L::kAtoms * kAtom);
      for (int at = 0; at < L::kAtoms; ++at)
        tma_load_2d(sm + L::kQ + at * kAtom, &a.tmap_q, q_full, h * a.head_stride + at * 64,
                    b * a.n_q + qt * kTcBQ);
      int j = 0;
      for (; j < nt; ++j) {
        const int s = j & 1;
        if (!mbar_wait(&kv_empty[s], ((j >> 1) & 1) ^ 1u, abort_flag, a.status, 11)) break;
        uint8_t* st = sm + L::kKV + s * L::kStage;
        mbar_arrive_expect_tx(&kv_full[s], 2 * L::kAtoms * kAtom);
        const int row = b * a.n_kv + j * kTcBK;
        for (int at = 0; at < L::kAtoms; ++at) {
          tma_load_2d(st + at * kAtom, &a.tmap_k, &kv_full[s], h * a.head_stride + at * 64, row);
          tma_load_2d(st + (L::kAtoms + at) * kAtom, &a.tmap_v, &kv_full[s], h * a.head_stride + at * 64, row);
        }
      }
      if (*abort_flag) {
        mbar_drain(q_full, 0);
        for (int i = (j > 2 ? j - 2 : 0); i < j; ++i) mbar_drain(&kv_full[i & 1], (i >> 1) & 1);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc_qk = umma_idesc_f16(kTcBQ, kTcBK);
      const uint32_t idesc_pv = umma_idesc_f16_bmn(kTcBQ, DH);
      bool ok = mbar_wait(q_full, 0, abort_flag, a.status, 12);
      auto issue_qk = [&](int j) -> bool {
        const int s = j & 1;
        const uint32_t ph = (j >> 1) & 1;
        if (!mbar_wait(&kv_full[s], ph, abort_flag, a.status, 13)) return false;
        if (!mbar_wait(&s_free[s], ph ^ 1u, abort_flag, a.status, 14)) return false;
        tc_fence_after();
        const uint32_t qa = smem_u32(sm + L::kQ);
        const uint32_t ka = smem_u32(sm + L::kKV + s * L::kStage);
#pragma unroll
        for (int ks = 0; ks < DH / 16; ++ks) {
          const uint32_t off = (ks >> 2) * kAtom + (ks & 3) * 32;
          umma_f16(tmem + L::kTmemS + s * kTcBK, smem_desc_sw128(qa + off), smem_desc_sw128(ka + off),
                   idesc_qk, ks > 0 ? 1u : 0u);
        }
        umma_commit(&s_full[s]);
        return true;
      };
      if (ok) ok = issue_qk(0);
      for (int j = 0; j < nt && ok; ++j) {
        if (j + 1 < nt && !(ok = issue_qk(j + 1))) break;
        const int s = j & 1;
        if (!(ok = mbar_wait(&p_full[s], (j >> 1) & 1, abort_flag, a.status, 15))) break;
        tc_fence_after();
        const uint32_t pa = smem_u32(sm + L::kP + s * L::kPBuf);
        const uint32_t va = smem_u32(sm + L::kKV + s * L::kStage + L::kAtoms * kAtom);
#pragma unroll
        for (int ks = 0; ks < kTcBK / 16; ++ks) {
          const uint64_t ad = smem_desc_sw128(pa + (ks >> 2) * kAtom + (ks & 3) * 32);
          const uint64_t bd = smem_desc_sw128_mn(va + ks * 2048, kAtom, 1024);
          umma_f16(tmem + L::kTmemO, ad, bd, idesc_pv, (j > 0 || ks > 0) ? 1u : 0u);
        }
        umma_commit(&kv_empty[s]);
        umma_commit(&o_done[s]);
      }
      umma_commit(drain);
      mbar_drain(drain, 0);
    }
  } else {
    const int q = warp & 3;
    const int row = q * 32 + lane;
    const uint32_t lane_base = static_cast<uint32_t>(q * 32) << 16;
    float m2 = -INFINITY, l = 0.f;
    bool ok = true;
    uint32_t r[kTcBK];
    for (int j = 0; j < nt; ++j) {
      const int s = j & 1;
      if (!(ok = warp_wait_bar(&s_full[s], (j >> 1) & 1, abort_flag, a.status, 16))) break;
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < kTcBK / 16; ++c) tmem_ld16(tmem + lane_base + L::kTmemS + s * kTcBK + 16 * c, r + 16 * c);
#pragma unroll
      for (int c = 0; c < kTcBK / 16; ++c) tmem_ld_wait16(r + 16 * c);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&s_free[s]);
      const int kb = j * kTcBK;
      // scores in log2 units; 8 independent max chains (one softmax warp per SM
      // sub-partition: the reductions are latency-, not throughput-bound)
      float mx[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) mx[i] = -INFINITY;
      if (kb + kTcBK <= a.n_kv) {
#pragma unroll
        for (int c = 0; c < kTcBK; ++c) {
          const float v = __uint_as_float(r[c]) * a.scale_log2;
          r[c] = __float_as_uint(v);
          mx[c & 7] = fmaxf(mx[c & 7], v);
        }
      } else {
#pragma unroll
        for (int c = 0; c < kTcBK; ++c) {
          const float v = (kb + c < a.n_kv) ? __uint_as_float(r[c]) * a.scale_log2 : -INFINITY;
          r[c] = __float_as_uint(v);
          mx[c & 7] = fmaxf(mx[c & 7], v);
        }
      }
      const float mt = fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])),
                             fmaxf(fmaxf(mx[4], mx[5]), fmaxf(mx[6], mx[7])));
      if (j == 0) {
        m2 = mt;
      } else if (__any_sync(0xffffffffu, mt > m2 + kRescaleLog2)) {
        // Warp-uniform branch (the TMEM loads and stores below are .sync.aligned): every
        // lane moves its reference to max(m2, mt), which keeps O / l exact.  O must hold
        // PV_{j-1} complete before it is rescaled.
        if (!(ok = warp_wait_bar(&o_done[(j - 1) & 1], ((j - 1) >> 1) & 1, abort_flag, a.status, 17))) break;
        tc_fence_after();
        const float mnew = fmaxf(m2, mt);
        const float corr = exp2f(m2 - mnew);
        uint32_t o16[16];
#pragma unroll
        for (int c = 0; c < DH / 16; ++c) {
          tmem_ld16(tmem + lane_base + L::kTmemO + 16 * c, o16);
          tmem_ld_wait16(o16);
#pragma unroll
          for (int i = 0; i < 16; ++i) o16[i] = __float_as_uint(__uint_as_float(o16[i]) * corr);
          tmem_st16(tmem + lane_base + L::kTmemO + 16 * c, o16);
        }
        tmem_st_wait();
        tc_fence_before();
        l *= corr;
        m2 = mnew;
      }
      // P buffer s was last read by PV_{j-2}
      if (j >= 2 && !(ok = warp_wait_bar(&o_done[s], ((j - 2) >> 1) & 1, abort_flag, a.status, 18))) break;
      uint8_t* pbuf = sm + L::kP + s * L::kPBuf;
      float ls[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) ls[i] = 0.f;
#pragma unroll
      for (int cc = 0; cc < kTcBK / 8; ++cc) {
        float p8[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          p8[i] = exp2f(__uint_as_float(r[cc * 8 + i]) - m2);
          ls[i] += p8[i];
        }
        uint8_t* dst = pbuf + (cc >> 3) * kAtom + row * 128 + ((((cc & 7) ^ (row & 7))) << 4);
        *reinterpret_cast<uint4*>(dst) = pack_f16x8(p8);
      }
      l += ((ls[0] + ls[1]) + (ls[2] + ls[3])) + ((ls[4] + ls[5]) + (ls[6] + ls[7]));
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_full[s]);
    }
    if (ok && warp_wait_bar(&o_done[(nt - 1) & 1], ((nt - 1) >> 1) & 1, abort_flag, a.status, 19)) {
      tc_fence_after();
      const float inv = 1.f / l;
      const int qrow = qt * kTcBQ + row;
      f16* orow = a.o + (static_cast<int64_t>(b) * a.n_q + qrow) * a.ldo + h * DH;
      uint32_t o16[16];
#pragma unroll
      for (int c = 0; c < DH / 16; ++c) {
        tmem_ld16(tmem + lane_base + L::kTmemO + 16 * c, o16);
        tmem_ld_wait16(o16);
        float f[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) f[i] = __uint_as_float(o16[i]) * inv;
        if (qrow < a.n_q) {
          reinterpret_cast<uint4*>(orow + 16 * c)[0] = pack_f16x8(f);
          reinterpret_cast<uint4*>(orow + 16 * c)[1] = pack_f16x8(f + 8);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem, 512);
  }
}

// ----------------------------------------------------------------------------
// attn_pp_kernel: two query tiles per CTA, ping-pong between two softmax warpgroups.
//
// One CTA = 256 queries (tiles 0 and 1) of one (sample, head); K/V tiles of 128 keys, shared
// by both query tiles, through a 2-stage TMA ring in which K and V have their own barriers: the
// K of tile j + 2 is fetched once S_1(j) has read K(j), not only after P V_1(j) (with one
// barrier for both, S_0(j + 1) waited 600 to 800 of the 3300 clocks of a key tile for it at d_h
// 128).  TMEM holds S_0, S_1 (128 fp32 columns each) and O_0, O_1 (d_h columns each).  Warps 2-5 run the softmax of tile 0, warps 6-9 of
// tile 1: each reads its S from TMEM (a max pass, then an exp pass), writes P as fp16 pairs
// over the first 64 columns of the same S, and the MMA warp computes O_t += P_t V from
// Tensor Memory (A operand in TMEM), so P needs no shared memory.  The MMA warp issues, per
// key tile j: PV_0(j), S_0(j+1), PV_1(j), S_1(j+1): while one warpgroup runs its softmax,
// the tensor cores work on the other tile.  tcgen05.mma operations of one thread run in
// issue order, so S_t(j+1) overwrites P_t(j) only after PV_t(j) has read it.
// ----------------------------------------------------------------------------
constexpr int kPpThreads = 320;
constexpr int kPpBQ = 256;

// d_h 64 / 128: every 128-row operand tile is d_h / 64 atoms of 64 columns (128-byte swizzle).
// d_h 72: the input heads are padded to 80 columns (columns 72..79 of Q zero), and a tile is
// one 64-column atom plus one 16-column atom (32-byte swizzle); Q K^T runs K = 80 (five
// K = 16 steps), P V runs as an N = 64 and an N = 16 instruction, O keeps 80 TMEM columns of
// which the first 72 are stored.
constexpr int kAtom32 = 128 * 16 * 2;  // 128 rows x 16 fp16: one 32-byte-swizzle column block

template <int DH>
struct PpLayout {
  static constexpr bool kPad = DH == 72;
  static constexpr int kA64 = DH / 64;                // 64-column atoms per tile
  static constexpr int kA16 = kPad ? 1 : 0;           // 16-column atoms per tile
  static constexpr int kDP = 64 * kA64 + 16 * kA16;   // head width the MMAs see
  static constexpr int kTile = kA64 * kAtom + kA16 * kAtom32;
  static constexpr int kQ = 0;                        // Q tile t at kQ + t kTile
  static constexpr int kKV = 2 * kTile;               // stage s: the K tile, then the V tile
  static constexpr int kStage = 2 * kTile;
  static constexpr int kBar = kKV + 2 * kStage;
  static constexpr int kBytes = kBar + 256 + 1024;
  static constexpr uint32_t kTmemS = 0;               // S_t at columns 128 t
  static constexpr uint32_t kTmemO = 256;             // O_t at columns 256 + kDP t
  static_assert(kBytes <= 232448, "shared memory");
  static_assert(kTmemO + 2 * kDP <= 512, "tensor memory");
};

template <int DH>
__global__ void __launch_bounds__(kPpThreads, 1) attn_pp_kernel(const __grid_constant__ AttnTcArgs a) {
  using L = PpLayout<DH>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + L::kBar);
  uint64_t* q_full = bars;
  uint64_t* k_full = bars + 1;
  uint64_t* k_empty = bars + 3;
  uint64_t* s_full = bars + 5;   // per query tile
  uint64_t* p_lo = bars + 7;     // per query tile, 4 warps arrive: P of the first 64 keys
  uint64_t* o_done = bars + 9;   // per query tile
  uint64_t* drain = bars + 11;
  uint64_t* p_hi = bars + 12;    // ... and of the other 64
  uint64_t* v_full = bars + 14;
  uint64_t* v_empty = bars + 16;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 18);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qt = blockIdx.x, bh = blockIdx.y;
  const int b = bh / a.n_heads, h = bh % a.n_heads;
  const int nt = (a.n_kv + kTcBK - 1) / kTcBK;
  // the second query tile of the last pair may hold no query (n_q % 256 in (0, 128], e.g. 258
  // tokens): that CTA then runs tile 0 alone (CTA-uniform)
  const bool two = (2 * qt + 1) * kTcBQ < a.n_q;

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&k_full[i], 1);
      mbar_init(&k_empty[i], 1);
      mbar_init(&v_full[i], 1);
      mbar_init(&v_empty[i], 1);
      mbar_init(&s_full[i], 1);
      mbar_init(&p_lo[i], 4);
      mbar_init(&p_hi[i], 4);
      mbar_init(&o_done[i], 1);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&a.tmap_q);
    tma_prefetch_desc(&a.tmap_k);
    tma_prefetch_desc(&a.tmap_v);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait_and_trigger();  // the prologue above touched only shared memory and TMEM
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    const bool lead = elect_one();
    const uint32_t sm0 = smem_u32(sm), k_full0 = smem_u32(k_full), k_empty0 = smem_u32(k_empty);
    const uint32_t v_full0 = smem_u32(v_full), v_empty0 = smem_u32(v_empty);
    const int col0 = h * a.head_stride;
    // one 128-row operand tile: its 64-column atoms, then (d_h 72) its 16-column atom
    auto load_tile = [&](uint32_t dst, const CUtensorMap* m64, const CUtensorMap* m16, uint32_t bar, int row) {
      for (int at = 0; at < L::kA64; ++at) tma_load_2d_at(dst + at * kAtom, m64, bar, col0 + at * 64, row);
      if (L::kPad) tma_load_2d_at(dst + L::kA64 * kAtom, m16, bar, col0 + 64, row);
    };
    if (lead) {
      const uint32_t bar = smem_u32(q_full);
      mbar_arrive_expect_tx_at(bar, (two ? 2 : 1) * L::kTile);
      for (int t = 0; t < (two ? 2 : 1); ++t)
        load_tile(sm0 + L::kQ + t * L::kTile, &a.tmap_q, &a.tmap_q16, bar, b * a.n_q + (2 * qt + t) * kTcBQ);
    }
    int j = 0;
    for (; j < nt; ++j) {
      const int s = j & 1;
      const uint32_t ph = ((j >> 1) & 1) ^ 1u, st = sm0 + L::kKV + s * L::kStage;
      const int row = b * a.n_kv + j * kTcBK;
      if (!mbar_wait_warp(k_empty0 + 8 * s, ph, abort_flag, a.status, 21)) break;
      if (lead) {
        mbar_arrive_expect_tx_at(k_full0 + 8 * s, L::kTile);
        load_tile(st, &a.tmap_k, &a.tmap_k16, k_full0 + 8 * s, row);
      }
      if (!mbar_wait_warp(v_empty0 + 8 * s, ph, abort_flag, a.status, 20)) break;
      if (lead) {
        mbar_arrive_expect_tx_at(v_full0 + 8 * s, L::kTile);
        load_tile(st + L::kTile, &a.tmap_v, &a.tmap_v16, v_full0 + 8 * s, row);
      }
    }
    if (lead && *abort_flag) {
      mbar_drain(q_full, 0);
      // (a K tile whose V tile was not asked for any more is the j-th)
      for (int i = (j > 2 ? j - 2 : 0); i < j; ++i) {
        mbar_drain(&k_full[i & 1], (i >> 1) & 1);
        mbar_drain(&v_full[i & 1], (i >> 1) & 1);
      }
      if (j < nt) mbar_drain(&k_full[j & 1], (j >> 1) & 1);
    }
  } else if (warp == 1) {
    // The whole warp runs the loop, one elected lane issues, and every operand of an MMA is a
    // warp-uniform base plus a constant: a single divergent thread that built each descriptor
    // took about 140 clocks per MMA, twice what a 128 x 128 x 16 MMA takes to run.
    const bool lead = elect_one();
    constexpr uint32_t idesc_qk = umma_idesc_f16(kTcBQ, kTcBK);
    constexpr uint32_t idesc_pv = umma_idesc_f16_bmn(kTcBQ, 64 * L::kA64);
    constexpr uint32_t idesc_pv16 = umma_idesc_f16_bmn(kTcBQ, 16);
    const uint32_t sm0 = smem_u32(sm), k_full0 = smem_u32(k_full), k_empty0 = smem_u32(k_empty);
    const uint32_t v_full0 = smem_u32(v_full), v_empty0 = smem_u32(v_empty);
    const uint32_t s_full0 = smem_u32(s_full), p_lo0 = smem_u32(p_lo), p_hi0 = smem_u32(p_hi), o_done0 = smem_u32(o_done);
    const uint64_t dq = smem_desc_sw128(sm0 + L::kQ), dk = smem_desc_sw128(sm0 + L::kKV);
    const uint64_t dv = smem_desc_sw128_mn(sm0 + L::kKV + L::kTile, kAtom, 1024);
    const uint64_t dq16 = smem_desc_sw32(sm0 + L::kQ + L::kA64 * kAtom);
    const uint64_t dk16 = smem_desc_sw32(sm0 + L::kKV + L::kA64 * kAtom);
    const uint64_t dv16 = smem_desc_sw32_mn(sm0 + L::kKV + L::kTile + L::kA64 * kAtom, kAtom32, 256);
    constexpr uint64_t kTileU = L::kTile >> 4, kStageU = L::kStage >> 4;  // in descriptor units of 16 bytes
    bool ok = mbar_wait_warp(smem_u32(q_full), 0, abort_flag, a.status, 22);
    auto issue_qk = [&](int t, int s) {
      if (!lead) return;
      const uint32_t d = tmem + L::kTmemS + t * kTcBK;
      const uint64_t qa = dq + t * kTileU, ka = dk + s * kStageU;
#pragma unroll
      for (int ks = 0; ks < 4 * L::kA64; ++ks) {
        const uint64_t off = ((ks >> 2) * kAtom + (ks & 3) * 32) >> 4;
        umma_f16(d, qa + off, ka + off, idesc_qk, ks > 0 ? 1u : 0u);
      }
      if (L::kPad)  // head columns 64..79 (Q's 72..79 are zero)
        umma_f16(d, dq16 + t * kTileU, dk16 + s * kStageU, idesc_qk, 1u);
      umma_commit_at(s_full0 + 8 * t);
    };
    // O_t (+)= P_t V over the 64 keys of one half, as soon as their P is there
    auto pv_half = [&](int t, int s, int half, uint32_t accumulate) {
      if (!lead) return;
      const uint32_t pa = tmem + L::kTmemS + t * kTcBK, d = tmem + L::kTmemO + t * L::kDP;
      const uint64_t va = dv + s * kStageU, va16 = dv16 + s * kStageU;
#pragma unroll
      for (int i = 0; i < kTcBK / 32; ++i) {
        const int ks = half * (kTcBK / 32) + i;
        umma_f16_ts(d, pa + 8 * ks, va + ks * (2048 >> 4), idesc_pv, i > 0 ? 1u : accumulate);
        if (L::kPad)  // O columns 64..79 from the 16-column V atom (8-key-row groups 256 B apart)
          umma_f16_ts(d + 64 * L::kA64, pa + 8 * ks, va16 + ks * (512 >> 4), idesc_pv16, i > 0 ? 1u : accumulate);
      }
      if (half) umma_commit_at(o_done0 + 8 * t);
    };
    auto issue_pv = [&](int t, int s, uint32_t ph, uint32_t accumulate) -> bool {
      if (!mbar_wait_warp(p_lo0 + 8 * t, ph, abort_flag, a.status, 24 + 2 * t)) return false;
      tc_fence_after();
      pv_half(t, s, 0, accumulate);
      if (!mbar_wait_warp(p_hi0 + 8 * t, ph, abort_flag, a.status, 24 + 2 * t)) return false;
      tc_fence_after();
      pv_half(t, s, 1, 1u);
      return true;
    };
    if (ok && (ok = mbar_wait_warp(k_full0, 0, abort_flag, a.status, 23))) {
      tc_fence_after();
      issue_qk(0, 0);
      if (two) issue_qk(1, 0);
      if (lead) umma_commit_at(k_empty0);
    }
    for (int j = 0; j < nt && ok; ++j) {
      const int s = j & 1;
      const uint32_t ph = j & 1, acc = j > 0 ? 1u : 0u;
      if (!(ok = mbar_wait_warp(v_full0 + 8 * s, (j >> 1) & 1, abort_flag, a.status, 30))) break;
      if (!(ok = issue_pv(0, s, ph, acc))) break;
      if (j + 1 < nt) {
        if (!(ok = mbar_wait_warp(k_full0 + 8 * (s ^ 1), ((j + 1) >> 1) & 1, abort_flag, a.status, 25))) break;
        tc_fence_after();
        issue_qk(0, s ^ 1);
      }
      if (two && !(ok = issue_pv(1, s, ph, acc))) break;
      if (lead) umma_commit_at(v_empty0 + 8 * s);
      if (j + 1 < nt) {
        if (two) issue_qk(1, s ^ 1);
        if (lead) umma_commit_at(k_empty0 + 8 * (s ^ 1));
      }
    }
    if (lead) {
      umma_commit(drain);
      mbar_drain(drain, 0);
    }
  } else {
    const int t = (warp - 2) >> 2;   // query tile of this warpgroup
    const int q = warp & 3;          // TMEM lane quarter
    const int row = q * 32 + lane;
    const uint32_t lane_base = static_cast<uint32_t>(q * 32) << 16;
    const uint32_t s_col = tmem + lane_base + L::kTmemS + t * kTcBK;
    const uint32_t o_col = tmem + lane_base + L::kTmemO + t * L::kDP;
    float m2 = -INFINITY, l = 0.f;
    bool ok = t == 0 || two;  // the warpgroup of an empty second tile has nothing to do
    uint32_t r[kTcBK];
    for (int j = 0; j < nt && ok; ++j) {
      if (!(ok = mbar_wait_warp(smem_u32(&s_full[t]), j & 1, abort_flag, a.status, 27))) break;
      tc_fence_after();
      const int kb = j * kTcBK;
      const int nvalid = min(a.n_kv - kb, kTcBK);  // keys of this tile (the rest are masked)
      // the whole S row in registers, one TMEM round trip
#pragma unroll
      for (int c = 0; c < kTcBK; c += 16) tmem_ld16(s_col + c, r + c);
#pragma unroll
      for (int c = 0; c < kTcBK; c += 16) tmem_ld_wait16(r + c);
      if (nvalid < kTcBK) {  // masked keys score -inf (P = 0)
#pragma unroll
        for (int c = 0; c < kTcBK; ++c)
          if (c >= nvalid) r[c] = __float_as_uint(-INFINITY);
      }
      // the row maximum of the raw scores (scale > 0 commutes with max), then log2 units
      const float mt = a.scale_log2 * row_max<kTcBK>(r);
      if (j == 0) {
        m2 = mt;
      } else if (__any_sync(0xffffffffu, mt > m2 + kRescaleLog2)) {
        // warp-uniform (the TMEM accesses are .sync.aligned); O_t must hold PV_t(j-1)
        if (!(ok = mbar_wait_warp(smem_u32(&o_done[t]), (j - 1) & 1, abort_flag, a.status, 28))) break;
        tc_fence_after();
        const float mnew = fmaxf(m2, mt);
        const float corr = exp2f(m2 - mnew);
        uint32_t o16[16];
#pragma unroll 1
        for (int c = 0; c < L::kDP; c += 16) {
          tmem_ld16(o_col + c, o16);
          tmem_ld_wait16(o16);
#pragma unroll
          for (int i = 0; i < 16; ++i) o16[i] = __float_as_uint(__uint_as_float(o16[i]) * corr);
          tmem_st16(o_col + c, o16);
        }
        tmem_st_wait();
        l *= corr;
        m2 = mnew;
      }
      // P as fp16 pairs, stored over columns [0, 64) of this S (chunk c's 16 packed columns land on
      // scores already read); the MMA warp starts on the first 64 keys while the others follow
      const uint64_t scale2 = pack_f32x2(a.scale_log2, a.scale_log2), neg_m2 = pack_f32x2(-m2, -m2);
      uint64_t sum[4] = {0, 0, 0, 0};
#pragma unroll
      for (int half = 0; half < 2; ++half) {
#pragma unroll
        for (int c = 64 * half; c < 64 * half + 64; c += 32) {
          exp_pack32(r + c, scale2, neg_m2, sum);
          tmem_st16(s_col + c / 2, r + c);
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(half ? &p_hi[t] : &p_lo[t]);
      }
      l += sum_f32x2(add_f32x2(add_f32x2(sum[0], sum[1]), add_f32x2(sum[2], sum[3])));
    }
    if (ok && mbar_wait_warp(smem_u32(&o_done[t]), (nt - 1) & 1, abort_flag, a.status, 29)) {
      tc_fence_after();
      const float inv = 1.f / l;
      const int qrow = (2 * qt + t) * kTcBQ + row;
      f16* orow = a.o + (static_cast<int64_t>(b) * a.n_q + qrow) * a.ldo + h * DH;
#pragma unroll
      for (int c = 0; c < L::kDP; c += 16) {
        tmem_ld16(o_col + c, r);
        tmem_ld_wait16(r);
        float f[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) f[i] = __uint_as_float(r[i]) * inv;
        if (qrow < a.n_q) {
          reinterpret_cast<uint4*>(orow + c)[0] = pack_f16x8(f);
          if (c + 16 <= DH) reinterpret_cast<uint4*>(orow + c)[1] = pack_f16x8(f + 8);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem, 512);
  }
}

// ----------------------------------------------------------------------------
// attn_sm_kernel: one query tile per CTA, key tiles of 64, several CTAs per SM.
//
// A CTA of attn_pp_kernel holds an SM alone, so that with few key tiles its prologue, first
// loads, the chain of its tiles and the last stores are all exposed, and a second wave of a few
// CTAs costs a whole one.  Here one CTA = 128 queries with S (64 fp32 columns) and O in 128 (d_h
// 64) or 256 columns of TMEM and 50 to 100 KB of shared memory: 3 (d_h 64) or 2 CTAs share an SM
// and cover each other's latencies, ragged key counts waste at most 63 keys, and a warp whose 32
// queries do not exist skips its softmax.  P overwrites S as in attn_pp_kernel.
//
// The first reference of a row is its maximum over 128 keys, as in attn_pp_kernel: with that of
// 64 keys the largest probability of up to 128 keys was often not 1 but a rounded value above it
// (77 keys: 2.40e-4 from float64 instead of 2.29e-4).  The scores of the second tile are formed
// once more ahead of the loop, into O's columns, for their maxima alone.
// ----------------------------------------------------------------------------
constexpr int kSmThreads = 192;
constexpr int kSmBK = 64;

template <int DH>
struct SmLayout {
  static constexpr bool kPad = DH == 72;
  static constexpr int kA64 = DH / 64, kA16 = kPad ? 1 : 0;
  static constexpr int kDP = 64 * kA64 + 16 * kA16;   // head width the MMAs see
  static constexpr int kAtomKV = kSmBK * 128, kAtomKV32 = kSmBK * 32;
  static constexpr int kQBytes = kA64 * kAtom + kA16 * kAtom32;
  static constexpr int kTile = kA64 * kAtomKV + kA16 * kAtomKV32;
  static constexpr int kStage = 2 * kTile;            // the K tile, then the V tile
  static constexpr int kKV = kQBytes;
  static constexpr int kBar = kKV + 2 * kStage;
  static constexpr int kBytes = kBar + 128 + 1024;
  static constexpr int kTmemCols = kSmBK + kDP <= 128 ? 128 : 256;
  static constexpr int kBlocks = DH == 64 ? 3 : 2;    // per SM
  static constexpr uint32_t kTmemO = kSmBK;
  static_assert(kKV % 1024 == 0 && kTile % 1024 == 0 && kStage % 1024 == 0, "swizzle atoms");
  static_assert(kBlocks * (kBytes + 1024) <= 233472 && kBlocks * kTmemCols <= 512, "CTAs per SM");
};

template <int DH>
__global__ void __launch_bounds__(kSmThreads, SmLayout<DH>::kBlocks) attn_sm_kernel(const __grid_constant__ AttnTcArgs a) {
  using L = SmLayout<DH>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + L::kBar);
  uint64_t* q_full = bars;
  uint64_t* kv_full = bars + 1;
  uint64_t* kv_empty = bars + 3;
  uint64_t* s_full = bars + 5;
  uint64_t* p_full = bars + 6;
  uint64_t* o_done = bars + 7;
  uint64_t* drain = bars + 8;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 9);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qt = blockIdx.x, bh = blockIdx.y;
  const int b = bh / a.n_heads, h = bh % a.n_heads;
  const int nt = (a.n_kv + kSmBK - 1) / kSmBK;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&a.tmap_q);
    tma_prefetch_desc(&a.tmap_k);
    tma_prefetch_desc(&a.tmap_v);
    mbar_init(q_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&kv_full[i], 1);
      mbar_init(&kv_empty[i], 1);
    }
    mbar_init(s_full, 1);
    mbar_init(p_full, 4);
    mbar_init(o_done, 1);
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, L::kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait_and_trigger();  // the prologue above touched only shared memory and TMEM
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    const bool lead = elect_one();
    const uint32_t sm0 = smem_u32(sm), kv_full0 = smem_u32(kv_full), kv_empty0 = smem_u32(kv_empty);
    const int col0 = h * a.head_stride;
    if (lead) {
      const uint32_t bar = smem_u32(q_full);
      const int row = b * a.n_q + qt * kTcBQ;
      mbar_arrive_expect_tx_at(bar, L::kQBytes);
      for (int at = 0; at < L::kA64; ++at) tma_load_2d_at(sm0 + at * kAtom, &a.tmap_q, bar, col0 + at * 64, row);
      if (L::kPad) tma_load_2d_at(sm0 + L::kA64 * kAtom, &a.tmap_q16, bar, col0 + 64, row);
    }
    int j = 0;
    for (; j < nt; ++j) {
      const int s = j & 1;
      if (!mbar_wait_warp(kv_empty0 + 8 * s, ((j >> 1) & 1) ^ 1u, abort_flag, a.status, 51)) break;
      if (lead) {
        const uint32_t st = sm0 + L::kKV + s * L::kStage, bar = kv_full0 + 8 * s;
        const int row = b * a.n_kv + j * kSmBK;
        mbar_arrive_expect_tx_at(bar, 2 * L::kTile);
        for (int at = 0; at < L::kA64; ++at) tma_load_2d_at(st + at * L::kAtomKV, &a.tmap_k, bar, col0 + at * 64, row);
        if (L::kPad) tma_load_2d_at(st + L::kA64 * L::kAtomKV, &a.tmap_k16, bar, col0 + 64, row);
        for (int at = 0; at < L::kA64; ++at)
          tma_load_2d_at(st + L::kTile + at * L::kAtomKV, &a.tmap_v, bar, col0 + at * 64, row);
        if (L::kPad) tma_load_2d_at(st + L::kTile + L::kA64 * L::kAtomKV, &a.tmap_v16, bar, col0 + 64, row);
      }
    }
    if (lead && *abort_flag) {
      mbar_drain(q_full, 0);
      for (int i = (j > 2 ? j - 2 : 0); i < j; ++i) mbar_drain(&kv_full[i & 1], (i >> 1) & 1);
    }
  } else if (warp == 1) {
    const bool lead = elect_one();
    constexpr uint32_t idesc_qk = umma_idesc_f16(kTcBQ, kSmBK);
    constexpr uint32_t idesc_pv = umma_idesc_f16_bmn(kTcBQ, 64 * L::kA64);
    constexpr uint32_t idesc_pv16 = umma_idesc_f16_bmn(kTcBQ, 16);
    const uint32_t sm0 = smem_u32(sm), kv_full0 = smem_u32(kv_full), kv_empty0 = smem_u32(kv_empty);
    const uint64_t dq = smem_desc_sw128(sm0), dk = smem_desc_sw128(sm0 + L::kKV);
    const uint64_t dv = smem_desc_sw128_mn(sm0 + L::kKV + L::kTile, L::kAtomKV, 1024);
    const uint64_t dq16 = smem_desc_sw32(sm0 + L::kA64 * kAtom);
    const uint64_t dk16 = smem_desc_sw32(sm0 + L::kKV + L::kA64 * L::kAtomKV);
    const uint64_t dv16 = smem_desc_sw32_mn(sm0 + L::kKV + L::kTile + L::kA64 * L::kAtomKV, L::kAtomKV32, 256);
    constexpr uint64_t kStageU = L::kStage >> 4;
    auto issue_qk = [&](uint32_t d, int s) {
      if (!lead) return;
      const uint64_t ka = dk + s * kStageU;
#pragma unroll
      for (int ks = 0; ks < 4 * L::kA64; ++ks)
        umma_f16(d, dq + (((ks >> 2) * kAtom + (ks & 3) * 32) >> 4),
                 ka + (((ks >> 2) * L::kAtomKV + (ks & 3) * 32) >> 4), idesc_qk, ks > 0 ? 1u : 0u);
      if (L::kPad) umma_f16(d, dq16, dk16 + s * kStageU, idesc_qk, 1u);  // head columns 64..79
    };
    bool ok = mbar_wait_warp(smem_u32(q_full), 0, abort_flag, a.status, 52) &&
              mbar_wait_warp(kv_full0, 0, abort_flag, a.status, 53);
    if (ok && nt > 1) ok = mbar_wait_warp(kv_full0 + 8, 0, abort_flag, a.status, 53);
    if (ok) {
      tc_fence_after();
      issue_qk(tmem, 0);
      if (nt > 1) issue_qk(tmem + L::kTmemO, 1);  // for its row maxima; PV(0) overwrites it
      if (lead) umma_commit_at(smem_u32(s_full));
    }
    for (int j = 0; j < nt && ok; ++j) {
      const int s = j & 1;
      if (!(ok = mbar_wait_warp(smem_u32(p_full), j & 1, abort_flag, a.status, 54))) break;
      tc_fence_after();
      if (lead) {
        const uint64_t va = dv + s * kStageU, va16 = dv16 + s * kStageU;
        const uint32_t acc = j > 0 ? 1u : 0u;
#pragma unroll
        for (int ks = 0; ks < kSmBK / 16; ++ks) {
          umma_f16_ts(tmem + L::kTmemO, tmem + 8 * ks, va + ks * (2048 >> 4), idesc_pv, ks > 0 ? 1u : acc);
          if (L::kPad)  // O columns 64..79
            umma_f16_ts(tmem + L::kTmemO + 64 * L::kA64, tmem + 8 * ks, va16 + ks * (512 >> 4), idesc_pv16,
                        ks > 0 ? 1u : acc);
        }
        umma_commit_at(kv_empty0 + 8 * s);
        umma_commit_at(smem_u32(o_done));
      }
      if (j + 1 < nt) {
        if (!(ok = mbar_wait_warp(kv_full0 + 8 * (s ^ 1), ((j + 1) >> 1) & 1, abort_flag, a.status, 55))) break;
        tc_fence_after();
        issue_qk(tmem, s ^ 1);  // after PV(j) in issue order, which reads P where S goes
        if (lead) umma_commit_at(smem_u32(s_full));
      }
    }
    if (lead) {
      umma_commit(drain);
      mbar_drain(drain, 0);
    }
  } else {
    const int q = warp & 3;
    const int row = q * 32 + lane, qrow = qt * kTcBQ + row;
    const uint32_t s_col = tmem + (static_cast<uint32_t>(q * 32) << 16), o_col = s_col + L::kTmemO;
    const bool any = qt * kTcBQ + q * 32 < a.n_q;  // warp-uniform: some of its queries exist
    float m2 = -INFINITY, l = 0.f;
    bool ok = true;
    uint32_t r[kSmBK];
    // the scores of key tile j from TMEM column `col` into r, and their maximum in log2 units
    auto load_scores = [&](uint32_t col, int j) {
      const int nvalid = min(a.n_kv - j * kSmBK, kSmBK);  // keys of this tile (the rest are masked)
#pragma unroll
      for (int c = 0; c < kSmBK; c += 16) tmem_ld16(col + c, r + c);
#pragma unroll
      for (int c = 0; c < kSmBK; c += 16) tmem_ld_wait16(r + c);
      if (nvalid < kSmBK) {
#pragma unroll
        for (int c = 0; c < kSmBK; ++c)
          if (c >= nvalid) r[c] = __float_as_uint(-INFINITY);
      }
      return a.scale_log2 * row_max<kSmBK>(r);
    };
    for (int j = 0; j < nt && ok; ++j) {
      if (!(ok = mbar_wait_warp(smem_u32(s_full), j & 1, abort_flag, a.status, 56))) break;
      tc_fence_after();
      if (any) {
        if (j == 0 && nt > 1) m2 = load_scores(o_col, 1);
        const float mt = load_scores(s_col, j);
        if (j == 0) {
          m2 = fmaxf(m2, mt);
        } else if (__any_sync(0xffffffffu, mt > m2 + kRescaleLog2)) {
          // warp-uniform (the TMEM accesses are .sync.aligned); O must hold PV(j-1)
          if (!(ok = mbar_wait_warp(smem_u32(o_done), (j - 1) & 1, abort_flag, a.status, 57))) break;
          tc_fence_after();
          const float mnew = fmaxf(m2, mt);
          const float corr = exp2f(m2 - mnew);
          uint32_t o16[16];
#pragma unroll 1
          for (int c = 0; c < L::kDP; c += 16) {
            tmem_ld16(o_col + c, o16);
            tmem_ld_wait16(o16);
#pragma unroll
            for (int i = 0; i < 16; ++i) o16[i] = __float_as_uint(__uint_as_float(o16[i]) * corr);
            tmem_st16(o_col + c, o16);
          }
          tmem_st_wait();
          l *= corr;
          m2 = mnew;
        }
        const uint64_t scale2 = pack_f32x2(a.scale_log2, a.scale_log2), neg_m2 = pack_f32x2(-m2, -m2);
        uint64_t sum[4] = {0, 0, 0, 0};
#pragma unroll
        for (int c = 0; c < kSmBK; c += 32) {
          exp_pack32(r + c, scale2, neg_m2, sum);
          tmem_st16(s_col + c / 2, r + c);
        }
        l += sum_f32x2(add_f32x2(add_f32x2(sum[0], sum[1]), add_f32x2(sum[2], sum[3])));
        tmem_st_wait();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full);
    }
    if (ok && mbar_wait_warp(smem_u32(o_done), (nt - 1) & 1, abort_flag, a.status, 58) && any) {
      tc_fence_after();
      const float inv = 1.f / l;
      f16* orow = a.o + (static_cast<int64_t>(b) * a.n_q + qrow) * a.ldo + h * DH;
#pragma unroll
      for (int c = 0; c < L::kDP; c += 16) {
        tmem_ld16(o_col + c, r);
        tmem_ld_wait16(r);
        float f[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) f[i] = __uint_as_float(r[i]) * inv;
        if (qrow < a.n_q) {
          reinterpret_cast<uint4*>(orow + c)[0] = pack_f16x8(f);
          if (c + 16 <= DH) reinterpret_cast<uint4*>(orow + c)[1] = pack_f16x8(f + 8);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem, L::kTmemCols);
  }
}

template <int DH>
AttnTcArgs tc_args(const AttnPlan& plan) {
  const AttnParams& p = plan.p;
  AttnTcArgs a;
  memcpy(&a.tmap_q, &plan.tmap_q, sizeof(CUtensorMap));
  memcpy(&a.tmap_k, &plan.tmap_kv, sizeof(CUtensorMap));
  memcpy(&a.tmap_v, &plan.tmap_v, sizeof(CUtensorMap));
  memcpy(&a.tmap_q16, &plan.tmap_q16, sizeof(CUtensorMap));
  memcpy(&a.tmap_k16, &plan.tmap_k16, sizeof(CUtensorMap));
  memcpy(&a.tmap_v16, &plan.tmap_v16, sizeof(CUtensorMap));
  a.head_stride = p.head_stride > 0 ? p.head_stride : DH;
  a.o = p.o;
  a.ldo = p.ldo;
  a.n_q = p.n_q;
  a.n_kv = p.n_kv;
  a.n_heads = p.n_heads;
  a.scale_log2 = 1.4426950408889634f / sqrtf(static_cast<float>(DH));
  a.status = device_status_ptr();
  return a;
}

template <int DH>
cudaError_t launch_sm(const AttnPlan& plan, cudaStream_t s) {
  using L = SmLayout<DH>;
  static bool done[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(attn_sm_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         L::kBytes);
    if (e != cudaSuccess) return e;
    done[dev] = true;
  }
  dim3 grid((plan.p.n_q + kTcBQ - 1) / kTcBQ, plan.p.batch * plan.p.n_heads);
  return launch_k(attn_sm_kernel<DH>, grid, dim3(kSmThreads), L::kBytes, s, tc_args<DH>(plan));
}

template <int DH>
cudaError_t launch_pp(const AttnPlan& plan, cudaStream_t s) {
  using L = PpLayout<DH>;
  static bool done[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(attn_pp_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         L::kBytes);
    if (e != cudaSuccess) return e;
    done[dev] = true;
  }
  const AttnParams& p = plan.p;
  dim3 grid((p.n_q + kPpBQ - 1) / kPpBQ, p.batch * p.n_heads);
  return launch_k(attn_pp_kernel<DH>, grid, dim3(kPpThreads), L::kBytes, s, tc_args<DH>(plan));
}

template <int DH>
cudaError_t launch_tc(const AttnPlan& plan, cudaStream_t s) {
  using L = TcLayout<DH>;
  static bool done[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(attn_tc_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         L::kBytes);
    if (e != cudaSuccess) return e;
    done[dev] = true;
  }
  const AttnParams& p = plan.p;
  AttnTcArgs a;
  memcpy(&a.tmap_q, &plan.tmap_q, sizeof(CUtensorMap));
  memcpy(&a.tmap_k, &plan.tmap_kv, sizeof(CUtensorMap));
  memcpy(&a.tmap_v, &plan.tmap_v, sizeof(CUtensorMap));
  a.head_stride = p.head_stride > 0 ? p.head_stride : DH;
  a.o = p.o;
  a.ldo = p.ldo;
  a.n_q = p.n_q;
  a.n_kv = p.n_kv;
  a.n_heads = p.n_heads;
  a.scale_log2 = 1.4426950408889634f / sqrtf(static_cast<float>(DH));
  a.status = device_status_ptr();
  dim3 grid((p.n_q + kTcBQ - 1) / kTcBQ, p.batch * p.n_heads);
  return launch_k(attn_tc_kernel<DH>, grid, dim3(kTcThreads), L::kBytes, s, a);
}

template <int DH, int DP>
cudaError_t launch_dh(const AttnParams& p, cudaStream_t s) {
  constexpr int kPitch = DP + 8;
  const int smem = (kBQ + 4 * kBKV) * kPitch * 2;
  static bool done[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(attn_kernel<DH, DP>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    done[dev] = true;
  }
  dim3 grid((p.n_q + kBQ - 1) / kBQ, p.batch * p.n_heads);
  return launch_k(attn_kernel<DH, DP>, grid, dim3(kWarps * 32), static_cast<size_t>(smem), s, p);
}

}  // namespace

int attn_check(const AttnParams& p, const char** why) {
  if (!p.q || !p.k || !p.v || !p.o || p.batch <= 0 || p.n_q <= 0 || p.n_kv <= 0 ||
      p.n_heads <= 0) {
    *why = "attention: null pointer or empty shape";
    return -1;
  }
  if (!(p.d_head == 64 || p.d_head == 72 || p.d_head == 128)) {
    *why = "attention: d_head must be 64, 72 or 128";
    return -2;
  }
  if ((p.ldq % 8) || (p.ldkv % 8) || (p.ldo % 8) ||
      ((reinterpret_cast<uintptr_t>(p.q) | reinterpret_cast<uintptr_t>(p.k) |
        reinterpret_cast<uintptr_t>(p.v) | reinterpret_cast<uintptr_t>(p.o)) & 15u)) {
    *why = "attention: leading dimensions must be multiples of 8, pointers 16-byte aligned";
    return -2;
  }
  if (p.batch * p.n_heads > 65535) {
    *why = "attention: batch * heads exceeds the grid limit";
    return -2;
  }
  if (p.head_stride != 0 && (p.head_stride < p.d_head || p.head_stride % 8)) {
    *why = "attention: head_stride must be >= d_head and a multiple of 8";
    return -2;
  }
  const int hs = p.head_stride > 0 ? p.head_stride : p.d_head;
  if (p.ldq < (p.n_heads - 1) * hs + p.d_head || p.ldkv < (p.n_heads - 1) * hs + p.d_head) {
    *why = "attention: ldq / ldkv smaller than the heads' columns";
    return -2;
  }
  return 0;
}

// Whether attn_sm_kernel runs this shape faster than attn_pp_kernel, by the time of each in us: a
// pair CTA holds an SM for a fixed part (more where it has both query tiles) and 1.1 to 1.4 us per
// 128 keys; a CTA of attn_sm_kernel takes a fixed part (more where the first reference looks at a
// second key tile) and 0.8 to 1 us per 64 keys by itself, and the SM 0.5 (d_h 64), 0.6 or 0.8 for one
// of several.  Fitted to 28 shapes, of which the chosen kernel is within 8% of the better one
// (measured us, pair / this kernel):
//   16 x 258 tokens, 16 heads of 64    24.9 / 17.3     2 x 1024, 20 heads of 64         24.2 / 20.6
//   2 x 1024 x 77 keys, 20 heads of 64 10.1 /  7.0     4 x 512, 16 heads of 64           8.6 / 11.2
//   1 x 333, 32 heads of 128            9.2 /  9.9     4 x 1024, 32 heads of 128        67.0 / 91.5
//   8 x 256, 16 heads of 72             7.8 /  8.7     2 x 136, 16 heads of 72           7.1 /  6.6
//   10 x 97 x 200 keys, 16 heads of 128 11.8 / 9.8     1 x 128, 8 heads of 64            4.3 /  4.8
bool attn_small(const AttnParams& p) {
  const double sms = num_sms(), heads = static_cast<double>(p.batch) * p.n_heads;
  const double pairs = std::ceil(p.n_q / 256.0) * heads, ctas = std::ceil(p.n_q / 128.0) * heads;
  const double nt = std::ceil(p.n_kv / 128.0), nt64 = std::ceil(p.n_kv / 64.0);
  const bool d64 = p.d_head == 64, d72 = p.d_head == 72, d128 = p.d_head == 128, two = p.n_q > kTcBQ;
  const double pair_fixed = d128 ? (two ? 4.9 : 4.5) : (two ? 3.8 : 3.0), pair_tile = d64 ? 1.14 : (d72 ? 1.3 : 1.42);
  const double sm_fixed = (d128 ? 4.0 : 2.0) + (nt64 > 1 ? 0.6 : 0.0), one_tile = d128 ? 0.83 : 1.0;
  const double sm_tile = d64 ? 0.52 : (d72 ? 0.6 : 0.8), slots = sms * (d64 ? 3 : 2);
  const double t_pair = std::ceil(pairs / sms) * (pair_fixed + nt * pair_tile);
  const double t_small = sm_fixed + nt64 * std::max(one_tile * std::ceil(ctas / slots), sm_tile * ctas / sms);
  return t_small < t_pair;
}

int attn_plan(AttnPlan& plan, const char** why) {
  const AttnParams& p = plan.p;
  int rc = attn_check(p, why);
  if (rc) return rc;
  const int hs = p.head_stride > 0 ? p.head_stride : p.d_head;
  // d_h 72 runs on tcgen05 only from a head-padded layout (>= 80 columns per head, Q's
  // columns 72..79 zero), with two query tiles per CTA
  const bool pad72 = p.d_head == 72 && hs >= 80;
  const bool tc_dh = p.d_head == 64 || p.d_head == 128 || (pad72 && p.impl != 2);
  plan.tc = (p.impl == 0 || p.impl == 2 || p.impl == 3) && tc_dh;
  if (!plan.tc) return 0;
  plan.pp = p.impl == 0 || p.impl == 3;
  plan.small = p.impl == 0 && attn_small(p);
  const int bk = plan.small ? kSmBK : kTcBK;
  const int cols = (p.n_heads - 1) * hs + (pad72 ? 80 : p.d_head);
  if (!make_tmap_f16(&plan.tmap_q, p.q, p.batch * p.n_q, cols, p.ldq, kTcBQ) ||
      !make_tmap_f16(&plan.tmap_kv, p.k, p.batch * p.n_kv, cols, p.ldkv, bk) ||
      !make_tmap_f16(&plan.tmap_v, p.v, p.batch * p.n_kv, cols, p.ldkv, bk)) {
    *why = "attention: cuTensorMapEncodeTiled failed";
    return -5;
  }
  if (pad72 && (!make_tmap_f16(&plan.tmap_q16, p.q, p.batch * p.n_q, cols, p.ldq, kTcBQ, 16) ||
                !make_tmap_f16(&plan.tmap_k16, p.k, p.batch * p.n_kv, cols, p.ldkv, bk, 16) ||
                !make_tmap_f16(&plan.tmap_v16, p.v, p.batch * p.n_kv, cols, p.ldkv, bk, 16))) {
    *why = "attention: cuTensorMapEncodeTiled failed";
    return -5;
  }
  return 0;
}

cudaError_t attn_launch(const AttnPlan& plan, cudaStream_t s) {
  const AttnParams& p = plan.p;
  if (plan.tc && plan.small)
    return p.d_head == 64 ? launch_sm<64>(plan, s) : (p.d_head == 72 ? launch_sm<72>(plan, s) : launch_sm<128>(plan, s));
  if (plan.tc && plan.pp)
    return p.d_head == 64 ? launch_pp<64>(plan, s) : (p.d_head == 72 ? launch_pp<72>(plan, s) : launch_pp<128>(plan, s));
  if (plan.tc) return p.d_head == 64 ? launch_tc<64>(plan, s) : launch_tc<128>(plan, s);
  switch (p.d_head) {
    case 64: return launch_dh<64, 64>(p, s);
    case 72: return launch_dh<72, 80>(p, s);
    default: return launch_dh<128, 128>(p, s);
  }
}

}  // namespace sgd
