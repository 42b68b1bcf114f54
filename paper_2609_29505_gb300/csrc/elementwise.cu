// Bandwidth-bound kernels of the scheduled step:
//   frozen_run   — Algorithm 2, frozen branch: h_{l,s} = h_{l-1,s} + Delta_{l, r_l(s)}
//                  for a run of consecutive frozen units in one read-modify-write of h
//                  (16-byte vectors: 8 fp32 of h, 8 fp16 of each cached update).
//   frozen_rows  — the same for models whose pre-norms are folded into the GEMMs, also
//                  writing fp16(h) and the partial row sums the next GEMM normalises with.
//   norm         — pre-norm of an active branch, fp32 residual in, fp16 GEMM operand out.
//   stem, gemv, head_small, copy_out, pack_f16 — the always-on parts around the
//                  scheduled units (input stage, conditioning, output head, U-ViT skip
//                  operands), Sec. 4.2: conditioning and skip features stay current.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "kernels.h"

namespace sgd {

namespace {

__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  float s = 0.f;
  const int nw = blockDim.x >> 5;
  for (int i = 0; i < nw; ++i) s += red[i];
  return s;
}

__device__ __forceinline__ void load_bf16x4(const bf16* p, float* f) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162* b = reinterpret_cast<const __nv_bfloat162*>(&u);
  float2 a = __bfloat1622float2(b[0]), c = __bfloat1622float2(b[1]);
  f[0] = a.x; f[1] = a.y; f[2] = c.x; f[3] = c.y;
}

// y = ((x - mean) * rstd) * g + b, then * (1 + scale) + shift (AdaLN), for the 4 columns
// 4 i .. 4 i + 3 of a row; sc / sh point at the row's sample's modulation (or are null).
template <class P>  // HeadParams (g, b: bf16 [d] or null)
__device__ __forceinline__ float4 norm_affine4(const P& p, int i, float4 v, float mean, float rstd,
                                               const float* sc, const float* sh) {
  float y[4] = {(v.x - mean) * rstd, (v.y - mean) * rstd, (v.z - mean) * rstd, (v.w - mean) * rstd};
  if (p.g) {
    float g[4];
    load_bf16x4(p.g + 4 * i, g);
#pragma unroll
    for (int k = 0; k < 4; ++k) y[k] *= g[k];
  }
  if (p.b) {
    float b[4];
    load_bf16x4(p.b + 4 * i, b);
#pragma unroll
    for (int k = 0; k < 4; ++k) y[k] += b[k];
  }
  if (sc) {
    const float4 s4 = *reinterpret_cast<const float4*>(sc + 4 * i);
    const float4 h4 = *reinterpret_cast<const float4*>(sh + 4 * i);
    y[0] = y[0] * (1.f + s4.x) + h4.x;
    y[1] = y[1] * (1.f + s4.y) + h4.y;
    y[2] = y[2] * (1.f + s4.z) + h4.z;
    y[3] = y[3] * (1.f + s4.w) + h4.w;
  }
  return make_float4(y[0], y[1], y[2], y[3]);
}

__device__ __forceinline__ void store_f16x4(f16* p, float4 v) { *reinterpret_cast<uint2*>(p) = pack_f16x4(v); }

// The affine part's parameters for the 4 columns 4 i .. of a row, read ahead of the row's
// statistics.  MODE: kGain bf16 gain and shift (either may be absent), no modulation; kMod an
// AdaLN modulation in 16-byte vectors, no gain or shift; kAny everything, the modulation as
// scalars at any alignment.
enum { kGain = 0, kMod = 1, kAny = 2 };
template <int MODE>
struct Affine4 {
  uint2 g, b;
  float4 sc, sh;
};
template <>
struct Affine4<kGain> {
  uint2 g, b;
};
template <>
struct Affine4<kMod> {
  float4 sc, sh;
};
template <int MODE>
__device__ __forceinline__ Affine4<MODE> load_affine4(const NormParams& p, int i, const float* sc, const float* sh) {
  Affine4<MODE> a;
  if constexpr (MODE != kMod) {
    if (p.g) a.g = __ldg(reinterpret_cast<const uint2*>(p.g + 4 * i));
    if (p.b) a.b = __ldg(reinterpret_cast<const uint2*>(p.b + 4 * i));
  }
  if constexpr (MODE == kMod) {
    a.sc = ld_f32x4(sc + 4 * i);
    a.sh = ld_f32x4(sh + 4 * i);
  }
  if constexpr (MODE == kAny) {
    if (sc) {
      a.sc = make_float4(sc[4 * i], sc[4 * i + 1], sc[4 * i + 2], sc[4 * i + 3]);
      a.sh = make_float4(sh[4 * i], sh[4 * i + 1], sh[4 * i + 2], sh[4 * i + 3]);
    }
  }
  return a;
}
__device__ __forceinline__ float4 bf16x4(uint2 u) {
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 c = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, c.x, c.y);
}
template <int MODE>
__device__ __forceinline__ float4 norm_apply4(const NormParams& p, const Affine4<MODE>& a, bool mod, float4 v,
                                              float mean, float rstd) {
  float4 y = make_float4((v.x - mean) * rstd, (v.y - mean) * rstd, (v.z - mean) * rstd, (v.w - mean) * rstd);
  if constexpr (MODE != kMod) {
    if (p.g) {
      const float4 g = bf16x4(a.g);
      y.x *= g.x; y.y *= g.y; y.z *= g.z; y.w *= g.w;
    }
    if (p.b) {
      const float4 b = bf16x4(a.b);
      y.x += b.x; y.y += b.y; y.z += b.z; y.w += b.w;
    }
  }
  if constexpr (MODE != kGain) {
    if (mod) {
      y.x = y.x * (1.f + a.sc.x) + a.sh.x;
      y.y = y.y * (1.f + a.sc.y) + a.sh.y;
      y.z = y.z * (1.f + a.sc.z) + a.sh.z;
      y.w = y.w * (1.f + a.sc.w) + a.sh.w;
    }
  }
  return y;
}

// Rows wider than 2048 (LLaDA's 4096): 256 threads per row, kWideVec float4 each, and a grid of
// a few blocks per SM that walk over the rows with the next row's loads in flight while the
// current one is reduced and stored.  One block per row left the loads of a block's only row
// exposed and a second, two-thirds full wave: 4096 x 4096 with h from DRAM 23.8 us, 18.7 so (5.4 of
// the 6.7 TB/s of a copy: one row ahead per block, with a barrier between its loads and its stores,
// is too little in flight); with h still in L2 17.0 and 15.9.
// Rows that fit in one wave of blocks get a block of 128 threads each (kPipe false).
constexpr int wide_threads(bool pipe) { return pipe ? 256 : 128; }  // d <= 4096: 4 or 8 float4 per thread
// per SM (with a gain alone the pipelined rows fit four blocks: 3% faster than three at 4096 x 4096)
constexpr int wide_blocks(int mode, bool pipe) { return pipe ? (mode == kGain ? 4 : 3) : 8; }
template <int MODE, bool kPipe>
__global__ void __launch_bounds__(wide_threads(kPipe), wide_blocks(MODE, kPipe)) norm_wide_kernel(const NormParams p) {
  constexpr int kThreads = wide_threads(kPipe), kVec = 1024 / kThreads;
  __shared__ float red[2][kThreads / 32];
  pdl_wait_and_trigger();
  const int nv = p.d >> 2, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float inv_d = 1.f / p.d;
  int flip = 0;
  auto block_total = [&](float v) {  // one barrier per reduction: the buffers alternate
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[flip][warp] = v;
    __syncthreads();
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < kThreads / 32; ++i) s += red[flip][i];
    flip ^= 1;
    return s;
  };
  float4 next[kVec];  // kPipe: the next row
  auto fetch = [&](int row) {
    const float4* hr = reinterpret_cast<const float4*>(p.h + static_cast<int64_t>(row) * p.d);
#pragma unroll
    for (int j = 0; j < kVec; ++j) {
      const int i = threadIdx.x + j * kThreads;
      next[j] = i < nv ? hr[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  if (static_cast<int>(blockIdx.x) < p.rows) fetch(blockIdx.x);
  for (int row = blockIdx.x; row < p.rows; row += gridDim.x) {
    float4 v[kVec];
#pragma unroll
    for (int j = 0; j < kVec; ++j) v[j] = next[j];
    const int64_t smp = p.scale ? row / p.rows_per_batch : 0;
    const float* sh = p.shift ? p.shift + smp * p.ld_mod : nullptr;
    const float* sc = p.scale ? p.scale + smp * p.ld_mod : nullptr;
    Affine4<MODE> af[kPipe ? kVec : 1];
    if (kPipe) {
#pragma unroll
      for (int j = 0; j < kVec; ++j) {
        const int i = threadIdx.x + j * kThreads;
        if (i < nv) af[kPipe ? j : 0] = load_affine4<MODE>(p, i, sc, sh);
      }
    }
    if (kPipe && row + gridDim.x < p.rows) fetch(row + gridDim.x);
    float mean = 0.f, sum = 0.f;
    if (p.kind != SGD_NORM_RMS) {
#pragma unroll
      for (int j = 0; j < kVec; ++j) sum += (v[j].x + v[j].y) + (v[j].z + v[j].w);
      mean = block_total(sum) * inv_d;
    }
    float sq = 0.f;
#pragma unroll
    for (int j = 0; j < kVec; ++j) {
      if (static_cast<int>(threadIdx.x) + j * kThreads < nv) {
        const float a = v[j].x - mean, b = v[j].y - mean, c = v[j].z - mean, d = v[j].w - mean;
        sq += (a * a + b * b) + (c * c + d * d);
      }
    }
    const float rstd = rsqrtf(block_total(sq) * inv_d + p.eps);
    f16* orow = p.out + static_cast<int64_t>(row) * p.d;
#pragma unroll
    for (int j = 0; j < kVec; ++j) {
      const int i = threadIdx.x + j * kThreads;
      if (i < nv) {
        const Affine4<MODE> a = kPipe ? af[kPipe ? j : 0] : load_affine4<MODE>(p, i, sc, sh);
        store_f16x4(orow + 4 * i, norm_apply4<MODE>(p, a, sc != nullptr, v[j], mean, rstd));
      }
    }
  }
}

// One warp per row (d <= 2048, NV float4 per lane): no block-wide reductions.  The row's
// modulation is read with the row, ahead of its statistics (reading them after, the
// modulation as scalars, took 6.2 us for 2048 x 1152 against the launch's ~2.5 us of traffic).
template <int NV, int MODE>
__global__ void __launch_bounds__(128, MODE != kGain ? 4 : (NV <= 8 ? 8 : 5)) norm_warp_kernel(const NormParams p) {
  pdl_wait_and_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * (blockDim.x >> 5) + warp;
  if (row >= p.rows) return;
  const int nv = p.d >> 2;
  const float4* hr = reinterpret_cast<const float4*>(p.h + static_cast<int64_t>(row) * p.d);
  const int64_t smp = p.scale ? row / p.rows_per_batch : 0;
  const float* sh = p.shift ? p.shift + smp * p.ld_mod : nullptr;
  const float* sc = p.scale ? p.scale + smp * p.ld_mod : nullptr;
  float4 v[NV];
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    const int i = lane + 32 * j;
    v[j] = i < nv ? hr[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // (a gain is the same for all rows, in L1 after the first; registers are better spent on rows)
  constexpr bool kAhead = NV <= 10 && MODE == kMod;
  Affine4<MODE> af[kAhead ? NV : 1];
  if (kAhead) {
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int i = lane + 32 * j;
      if (i < nv) af[kAhead ? j : 0] = load_affine4<MODE>(p, i, sc, sh);
    }
  }
  float sum = 0.f, sq = 0.f;
#pragma unroll
  for (int j = 0; j < NV; ++j) sum += (v[j].x + v[j].y) + (v[j].z + v[j].w);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const float mean = p.kind == SGD_NORM_RMS ? 0.f : sum / p.d;
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    if (lane + 32 * j < nv) {
      const float a = v[j].x - mean, b = v[j].y - mean, c = v[j].z - mean, d = v[j].w - mean;
      sq += (a * a + b * b) + (c * c + d * d);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  const float rstd = rsqrtf(sq / p.d + p.eps);
  f16* orow = p.out + static_cast<int64_t>(row) * p.d;
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    const int i = lane + 32 * j;
    if (i < nv) {
      const Affine4<MODE> a = kAhead ? af[kAhead ? j : 0] : load_affine4<MODE>(p, i, sc, sh);
      store_f16x4(orow + 4 * i, norm_apply4<MODE>(p, a, sc != nullptr, v[j], mean, rstd));
    }
  }
}

// Lagged drift of one group's input (App. B.1): each of kDriftBlocks blocks strides over
// float4s of h (two per iteration, to keep more loads in flight), accumulating (h - snap)^2
// and h^2 per thread in fp32, reduces them in a fixed tree and writes its pair; snap takes
// the current h for the next step.  The grid size is fixed, so the summation order (and
// the result) is the same on every run.
__device__ __forceinline__ void drift_acc(const float4 x, const float4 y, float& dd, float& hh) {
  const float a = x.x - y.x, b = x.y - y.y, c = x.z - y.z, d = x.w - y.w;
  dd += (a * a + b * b) + (c * c + d * d);
  hh += (x.x * x.x + x.y * x.y) + (x.z * x.z + x.w * x.w);
}

__global__ void __launch_bounds__(256) drift_kernel(const DriftParams p) {
  __shared__ float red[8];
  pdl_wait_and_trigger();
  const int64_t nv = p.n >> 2;
  const float4* h4 = reinterpret_cast<const float4*>(p.h);
  float4* s4 = reinterpret_cast<float4*>(p.snap);
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  float dd = 0.f, hh = 0.f;
  int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  for (; i + stride < nv; i += 2 * stride) {
    const float4 x0 = h4[i], y0 = s4[i], x1 = h4[i + stride], y1 = s4[i + stride];
    drift_acc(x0, y0, dd, hh);
    drift_acc(x1, y1, dd, hh);
    s4[i] = x0;
    s4[i + stride] = x1;
  }
  if (i < nv) {
    const float4 x = h4[i], y = s4[i];
    drift_acc(x, y, dd, hh);
    s4[i] = x;
  }
  dd = block_sum(dd, red);
  hh = block_sum(hh, red);
  if (threadIdx.x == 0) {
    p.partial[2 * blockIdx.x] = dd;
    p.partial[2 * blockIdx.x + 1] = hh;
  }
}

// One warp per group: lane l sums partials l, l + 32, ... in double, then a fixed xor tree
// combines the lanes (the order is the same on every run).
__global__ void drift_reduce_kernel(const float* partials, double* sums) {
  pdl_wait_and_trigger();
  const float* p = partials + static_cast<size_t>(blockIdx.x) * 2 * kDriftBlocks;
  double dd = 0.0, hh = 0.0;
  for (int b = threadIdx.x; b < kDriftBlocks; b += 32) {
    dd += static_cast<double>(p[2 * b]);
    hh += static_cast<double>(p[2 * b + 1]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    dd += __shfl_xor_sync(0xffffffffu, dd, o);
    hh += __shfl_xor_sync(0xffffffffu, hh, o);
  }
  if (threadIdx.x == 0) {
    sums[2 * blockIdx.x] = dd;
    sums[2 * blockIdx.x + 1] = hh;
  }
}

// Failure-path self-test: thread 0 waits, with the kernels' bounded wait, on an mbarrier
// whose phase nothing completes; after the wait limit it records `code` in the device
// status word and returns.  Used to test the timeout path without faulting the GPU.
__global__ void wait_selftest_kernel(int* status, int code) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_wait(&bar, 0, &abort_flag, status, code);
}

__global__ void __launch_bounds__(256) frozen_kernel(const __grid_constant__ FrozenParams p) {
  pdl_wait_and_trigger();
  const int64_t n8 = p.n >> 3;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n8; i += stride) {
    float4* hp = reinterpret_cast<float4*>(p.h) + 2 * i;
    const float4 a = hp[0], b = hp[1];
    float acc[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    for (int c = 0; c < p.n_caches; ++c) {
      const uint4 u = __ldcs(reinterpret_cast<const uint4*>(p.caches[c]) + i);
      float f[8];
      unpack_f16x8(u, f);
#pragma unroll
      for (int k = 0; k < 8; ++k) acc[k] += f[k];
    }
    hp[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    hp[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
  }
}

// Frozen run for models whose pre-norms are folded into the GEMMs: also the writer of h's
// fp16 copy and row sums.  Warp w of the grid takes chunk (row, ch) of kStatChunk columns;
// each lane handles 8 consecutive columns per 256-column step, adds the cached updates in
// cache order (the same fp32 arithmetic as frozen_kernel), stores h and fp16(h), and the
// warp reduces its sums with a fixed xor tree into stat slot ch.
__global__ void __launch_bounds__(256) frozen_rows_kernel(const __grid_constant__ FrozenParams p) {
  pdl_wait_and_trigger();
  const int nch = (p.d + kStatChunk - 1) / kStatChunk;
  const int64_t wid = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (wid >= static_cast<int64_t>(p.rows) * nch) return;
  const int lane = threadIdx.x & 31;
  const int row = static_cast<int>(wid / nch), ch = static_cast<int>(wid % nch);
  const int c1 = min(p.d, (ch + 1) * kStatChunk);
  float ss = 0.f, s1 = 0.f;
  for (int c = ch * kStatChunk + lane * 8; c < c1; c += 256) {
    const int64_t i = (static_cast<int64_t>(row) * p.d + c) >> 3;
    float4* hp = reinterpret_cast<float4*>(p.h) + 2 * i;
    const float4 a = hp[0], b = hp[1];
    float acc[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    for (int k = 0; k < p.n_caches; ++k) {
      const uint4 u = __ldcs(reinterpret_cast<const uint4*>(p.caches[k]) + i);
      float f[8];
      unpack_f16x8(u, f);
#pragma unroll
      for (int q = 0; q < 8; ++q) acc[q] += f[q];
    }
    if (p.n_caches) {
      hp[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      hp[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
    reinterpret_cast<uint4*>(p.h16)[i] = pack_f16x8(acc);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      ss = fmaf(acc[q], acc[q], ss);
      s1 += acc[q];
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
  }
  if (lane == 0) {
    p.stat[static_cast<int64_t>(ch) * p.rows + row] = ss;
    p.stat[static_cast<int64_t>(kStatSlots + ch) * p.rows + row] = s1;
  }
}

// Writes the step's I/O slot and its time embeddings sinusoid(t, dim)[c] = cos(t w_i) for c < half,
// sin(t w_{c-half}) otherwise, w_i = 10000^(-i / half) (a table in double, made at creation).  The
// cosine and sine are in double, at a few dozen results per clock for the whole GPU: formed here
// once per step instead of by every block (or element) that reads them.
__global__ void io_set_kernel(IoSlot* slot, const IoSlot v, const TimeEmb te) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *slot = v;
  if (i >= te.n) return;
  int dim = te.dim0, c = i;
  const double* w = te.w;
  if (c >= te.dim0) {
    c -= te.dim0;
    w += te.dim0 >> 1;
    dim = te.n - te.dim0;
  }
  const int half = dim >> 1;
  const double t = v.t;
  te.out[i] = static_cast<float>(c < half ? cos(t * w[c]) : sin(t * w[c - half]));
}

// The stems of arbitrary widths: one thread per element.
__global__ void stem_kernel(const StemParams p) {
  pdl_wait_and_trigger();
  const int64_t total = static_cast<int64_t>(p.batch) * p.n_tokens * p.d;
  const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const int c = static_cast<int>(idx % p.d);
  const int64_t r = idx / p.d;
  const int n = static_cast<int>(r % p.n_tokens);
  const int b = static_cast<int>(r / p.n_tokens);
  const IoSlot* s = p.slot;
  float v = 0.f;
  const int np = n - p.n_prefix;
  if (np < 0) {
    const int cls = min(max(s->class_ids[b], 0), p.n_classes - 1);
    v = (n == 0) ? p.time[c]
                 : __bfloat162float(p.class_emb[static_cast<int64_t>(cls) * p.d + c]);
  } else {
    const float* z = reinterpret_cast<const float*>(s->state) +
                     (static_cast<int64_t>(b) * (p.n_tokens - p.n_prefix) + np) * p.d_in;
    const bf16* w = p.w_stem + static_cast<int64_t>(c) * p.d_in;
    float acc = 0.f;
    for (int k = 0; k < p.d_in; ++k) acc = fmaf(z[k], __bfloat162float(w[k]), acc);
    v = acc;
  }
  v += __bfloat162float(p.pos[static_cast<int64_t>(n) * p.d + c]);
  p.h[idx] = v;
}

// The stems without a projection (d % 8 == 0), bound by writing h: thread (x, y) handles 8
// columns of every gridDim.y-th row in 16-byte vectors (4096 x 4096 embedding rows: 72 us with
// one element per thread).
__global__ void __launch_bounds__(128) stem_rows_kernel(const StemParams p) {
  pdl_wait_and_trigger();
  const int c0 = (blockIdx.x * blockDim.x + threadIdx.x) * 8;
  if (c0 >= p.d) return;
  const IoSlot* s = p.slot;
  const int rows = p.batch * p.n_tokens;
  float4 ta = make_float4(0.f, 0.f, 0.f, 0.f), tb = ta;
  if (p.kind == SGD_STEM_TIME_ADD) {
    ta = *reinterpret_cast<const float4*>(p.time + c0);
    tb = *reinterpret_cast<const float4*>(p.time + c0 + 4);
  }
  for (int r = blockIdx.y; r < rows; r += gridDim.y) {
    const int64_t at = static_cast<int64_t>(r) * p.d + c0;
    float4 a, b;
    if (p.kind == SGD_STEM_EMBED) {
      const int id = min(max(reinterpret_cast<const int32_t*>(s->state)[r], 0), p.vocab - 1);
      const uint4 u = __ldg(reinterpret_cast<const uint4*>(p.embed + static_cast<int64_t>(id) * p.d + c0));
      a = bf16x4(make_uint2(u.x, u.y));
      b = bf16x4(make_uint2(u.z, u.w));
    } else {
      const float4* z = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(s->state) + at);
      a = z[0];
      b = z[1];
      if (p.kind == SGD_STEM_TIME_ADD) {
        a.x += ta.x; a.y += ta.y; a.z += ta.z; a.w += ta.w;
        b.x += tb.x; b.y += tb.y; b.z += tb.z; b.w += tb.w;
      }
    }
    float4* h = reinterpret_cast<float4*>(p.h + at);
    h[0] = a;
    h[1] = b;
  }
}

// The patch stems (d_in % 8 == 0, d % 4 == 0), bound by writing h: a thread owns 4 channels, with
// their DIN-wide weight rows in registers, and a block walks over kPatchRows token rows whose
// patches it has put in shared memory (read by every thread alike).  One thread per (row, 4
// channels) read its 4 weight rows again for every row, 32 different lines per load: 22 us for
// 2048 x 1152.  Each channel's dot product is summed in k order as in stem_kernel.
constexpr int kPatchRows = 8;
template <int DIN>
__global__ void __launch_bounds__(128) stem_patch_kernel(const StemParams p) {
  __shared__ float4 zs[kPatchRows][DIN / 4];
  pdl_wait_and_trigger();
  const IoSlot* s = p.slot;
  const int col_blocks = ((p.d >> 2) + 127) / 128;  // in grid.x with the rows, which may be millions
  const int rows = p.batch * p.n_tokens, r0 = (blockIdx.x / col_blocks) * kPatchRows, nr = min(kPatchRows, rows - r0);
  const int n_in = p.n_tokens - p.n_prefix;
  for (int i = threadIdx.x; i < nr * (DIN / 4); i += blockDim.x) {
    const int k = i / (DIN / 4), r = r0 + k;
    const int n = r % p.n_tokens - p.n_prefix, b = r / p.n_tokens;
    if (n >= 0)
      zs[k][i % (DIN / 4)] = reinterpret_cast<const float4*>(s->state)[(static_cast<int64_t>(b) * n_in + n) * (DIN / 4) + i % (DIN / 4)];
  }
  const int c0 = ((blockIdx.x % col_blocks) * blockDim.x + threadIdx.x) * 4;
  const bool active = c0 < p.d;
  float w[4][DIN];
  if (active) {
    const uint4* wp = reinterpret_cast<const uint4*>(p.w_stem + static_cast<int64_t>(c0) * DIN);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int k8 = 0; k8 < DIN / 8; ++k8) unpack_bf16x8(__ldg(wp + q * (DIN / 8) + k8), &w[q][8 * k8]);
  }
  __syncthreads();
  if (!active) return;
  uint2 pos_next = __ldg(reinterpret_cast<const uint2*>(p.pos + static_cast<int64_t>(r0 % p.n_tokens) * p.d + c0));
#pragma unroll 1
  for (int k = 0; k < nr; ++k) {
    const int r = r0 + k, n = r % p.n_tokens, b = r / p.n_tokens;
    const float4 ps = bf16x4(pos_next);
    pos_next = __ldg(reinterpret_cast<const uint2*>(p.pos + static_cast<int64_t>((r + 1) % p.n_tokens) * p.d + c0));
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n < p.n_prefix) {
      const int cls = min(max(s->class_ids[b], 0), p.n_classes - 1);
      v = n == 0 ? *reinterpret_cast<const float4*>(p.time + c0)
                 : bf16x4(*reinterpret_cast<const uint2*>(p.class_emb + static_cast<int64_t>(cls) * p.d + c0));
    } else {
#pragma unroll
      for (int i = 0; i < DIN / 4; ++i) {
        const float4 z = zs[k][i];
        v.x = fmaf(z.w, w[0][4 * i + 3], fmaf(z.z, w[0][4 * i + 2], fmaf(z.y, w[0][4 * i + 1], fmaf(z.x, w[0][4 * i], v.x))));
        v.y = fmaf(z.w, w[1][4 * i + 3], fmaf(z.z, w[1][4 * i + 2], fmaf(z.y, w[1][4 * i + 1], fmaf(z.x, w[1][4 * i], v.y))));
        v.z = fmaf(z.w, w[2][4 * i + 3], fmaf(z.z, w[2][4 * i + 2], fmaf(z.y, w[2][4 * i + 1], fmaf(z.x, w[2][4 * i], v.z))));
        v.w = fmaf(z.w, w[3][4 * i + 3], fmaf(z.z, w[3][4 * i + 2], fmaf(z.y, w[3][4 * i + 1], fmaf(z.x, w[3][4 * i], v.w))));
      }
    }
    *reinterpret_cast<float4*>(p.h + static_cast<int64_t>(r) * p.d + c0) =
        make_float4(v.x + ps.x, v.y + ps.y, v.z + ps.z, v.w + ps.w);
  }
}

// Patch widths without an instantiation above (d_in % 8 == 0): one thread per (token row, 4
// channels), the row's patch and the 4 channels' weight rows read as 16-byte vectors.
__global__ void stem_patch_any_kernel(const StemParams p) {
  pdl_wait_and_trigger();
  const int d4 = p.d >> 2;
  const int64_t total = static_cast<int64_t>(p.batch) * p.n_tokens * d4;
  const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const int c0 = static_cast<int>(idx % d4) * 4;
  const int64_t r = idx / d4;
  const int n = static_cast<int>(r % p.n_tokens);
  const int b = static_cast<int>(r / p.n_tokens);
  const IoSlot* s = p.slot;
  float v[4];
  const int np = n - p.n_prefix;
  if (np < 0) {
    const int cls = min(max(s->class_ids[b], 0), p.n_classes - 1);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      v[q] = (n == 0) ? p.time[c0 + q]
                      : __bfloat162float(p.class_emb[static_cast<int64_t>(cls) * p.d + c0 + q]);
  } else {
    const float4* z = reinterpret_cast<const float4*>(
        reinterpret_cast<const float*>(s->state) + (static_cast<int64_t>(b) * (p.n_tokens - p.n_prefix) + np) * p.d_in);
    const uint4* w = reinterpret_cast<const uint4*>(p.w_stem + static_cast<int64_t>(c0) * p.d_in);
    const int w_ld = p.d_in >> 3;  // uint4 per weight row
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = 0.f;
    for (int k8 = 0; k8 < w_ld; ++k8) {
      const float4 za = z[2 * k8], zb = z[2 * k8 + 1];
      const float zf[8] = {za.x, za.y, za.z, za.w, zb.x, zb.y, zb.z, zb.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float wf[8];
        unpack_bf16x8(__ldg(w + q * w_ld + k8), wf);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[q] = fmaf(zf[e], wf[e], v[q]);
      }
    }
  }
  const uint2 pu = __ldg(reinterpret_cast<const uint2*>(p.pos + static_cast<int64_t>(n) * p.d + c0));
  const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&pu);
  const float2 p01 = __bfloat1622float2(pb[0]), p23 = __bfloat1622float2(pb[1]);
  reinterpret_cast<float4*>(p.h)[idx] = make_float4(v[0] + p01.x, v[1] + p01.y, v[2] + p23.x, v[3] + p23.y);
}

// out[r, j] = sum_k act(x[r, k]) W[j, k] for R <= RMAX rows (conditioning and AdaLN
// modulation: a few rows against a large weight, bound by reading W once).  The block stages
// x once in shared memory and then works through output items (32 consecutive columns of one
// segment) with a grid of at most two blocks per SM.  Each warp owns 4 columns of an item; a
// lane streams 16-byte chunks (8 k) of the 4 weight rows and reuses each x chunk across them.
// x is staged as two planes (k % 8 < 4, k % 8 >= 4) so that the lanes' 16-byte x loads are
// consecutive (no bank conflicts).  With 8 rows the warp's 4 x 8 partial sums are reduced by
// a transpose reduction (31 shuffles, lane l ends with value l) instead of 32 butterflies.
//
// The products are formed as pairs of even and odd k (fma.rn.f32x2, two fp32 fmas per
// instruction, both halves added at the end): with one fma per instruction and 8 rows the fma
// pipe came close to the weight stream's time.
// v[0..31] of every lane -> lane l returns the warp's sum of value l
__device__ __forceinline__ float transpose_reduce32(float* v, int lane) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    const bool upper = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float a = v[i], b = v[i + o];
      const float send = upper ? a : b;
      v[i] = (upper ? b : a) + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return v[0];
}

__device__ __forceinline__ void gemv_store(const GemvParams& p, float* out, int r, int j, float v) {
  if (p.add_class) {
    const int cls = min(max(p.slot->class_ids[r], 0), p.n_classes - 1);
    v += __bfloat162float(p.add_class[static_cast<int64_t>(cls) * p.N + j]);
  }
  if (p.add_vec) v += p.add_vec[j];
  out[static_cast<int64_t>(r) * p.ldo + j] = v;
  if (p.out_silu) p.out_silu[static_cast<int64_t>(r) * p.ldo + j] = silu_f(v);
}

// COLS columns per warp: 32 / RMAX with several rows, 4 with one; 1 where the columns are too few
// to fill the SMs otherwise (the conditioning MLP: 1152 columns, the head's modulation: 2304).
template <int RMAX, int COLS>
__global__ void __launch_bounds__(256) gemv_kernel(const GemvParams p) {
  extern __shared__ float xs[];  // [xrows][2 planes][K / 2]
  pdl_wait_and_trigger();
  const int xrows = p.ldx == 0 ? 1 : p.rows;
  const int K = p.K, half = K >> 1;
  // x[r][k] lives at r * K + (k & 4 ? half : 0) + (k >> 3) * 4 + (k & 3)
  {
    // float4 loads (K % 8 == 0, rows 16-byte aligned) in batches of 8 per thread, every load
    // of a batch issued before its first shared-memory store: x is a generic pointer that
    // the compiler cannot tell apart from xs, so a store in between would make each load
    // wait for the previous element's round trip
    const int k4 = K >> 2, n4 = xrows * k4;
    constexpr int kBatch = 8;
    for (int i0 = threadIdx.x; i0 < n4; i0 += kBatch * blockDim.x) {
      float4 v[kBatch];
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int i = i0 + j * blockDim.x;
        if (i < n4) {
          const int r = i / k4, k = (i - r * k4) << 2;
          v[j] = ld_f32x4(p.x + static_cast<int64_t>(r) * p.ldx + k);
        }
      }
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int i = i0 + j * blockDim.x;
        if (i < n4) {
          const int r = i / k4, k = (i - r * k4) << 2;
          float4 x = v[j];
          if (p.in_silu) {
            x.x = silu_f(x.x);
            x.y = silu_f(x.y);
            x.z = silu_f(x.z);
            x.w = silu_f(x.w);
          }
          *reinterpret_cast<float4*>(xs + r * K + ((k & 4) ? half : 0) + (k >> 3) * 4) = x;
        }
      }
    }
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kCols = COLS;
  constexpr int kItemCols = 8 * kCols;  // 8 warps
  const int per_seg = (p.N + kItemCols - 1) / kItemCols;
  const int n_items = per_seg * (p.n_seg > 0 ? p.n_seg : 1);
  for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
    const int seg = item / per_seg;
    const int j0 = (item - seg * per_seg) * kItemCols + warp * kCols;
    if (j0 >= p.N) continue;  // warp-uniform; no block-wide barrier follows
    const bf16* W = p.n_seg ? p.w_seg[seg] : p.W;
    float* out = p.n_seg ? p.out_seg[seg] : p.out;
    uint64_t acc2[kCols * RMAX];  // sums over even and odd k
#pragma unroll
    for (int i = 0; i < kCols * RMAX; ++i) acc2[i] = 0;
    // unrolled so that a warp's weight loads for several K steps are in flight together
#pragma unroll 4
    for (int k = lane * 8; k < K; k += 256) {
      uint4 w[kCols];  // columns past N repeat the last one, whose sums are then not stored
#pragma unroll
      for (int c = 0; c < kCols; ++c)
        w[c] = __ldg(reinterpret_cast<const uint4*>(W + static_cast<int64_t>(min(j0 + c, p.N - 1)) * K + k));
      const int xo = (k >> 3) * 4;
      uint64_t wf[kCols][4];
#pragma unroll
      for (int c = 0; c < kCols; ++c) {
        const uint32_t u[4] = {w[c].x, w[c].y, w[c].z, w[c].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) wf[c][q] = pack_f32x2(u[q] << 16, u[q] & 0xffff0000u);
      }
#pragma unroll
      for (int r = 0; r < RMAX; ++r) {
        if (r < xrows) {
          const ulonglong2 xa = *reinterpret_cast<const ulonglong2*>(xs + r * K + xo);
          const ulonglong2 xb = *reinterpret_cast<const ulonglong2*>(xs + r * K + half + xo);
          const uint64_t xv[4] = {xa.x, xa.y, xb.x, xb.y};
#pragma unroll
          for (int c = 0; c < kCols; ++c)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc2[c * RMAX + r] = fma_f32x2(wf[c][q], xv[q], acc2[c * RMAX + r]);
        }
      }
    }
    float acc[kCols * RMAX];
#pragma unroll
    for (int i = 0; i < kCols * RMAX; ++i) acc[i] = sum_f32x2(acc2[i]);
    if constexpr (kCols * RMAX == 8) {  // one column: lanes 4 i .. 4 i + 3 end with row i
#pragma unroll
      for (int o = 16; o >= 4; o >>= 1) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o / 4; ++i) {
          const float send = upper ? acc[i] : acc[i + o / 4];
          acc[i] = (upper ? acc[i + o / 4] : acc[i]) + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      float v = acc[0];
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      if ((lane & 3) == 0 && (lane >> 2) < p.rows) gemv_store(p, out, lane >> 2, j0, v);
    } else if constexpr (kCols * RMAX == 32) {
      // lane l: column j0 + l / RMAX, row l % RMAX
      const float v = transpose_reduce32(acc, lane);
      const int c = lane / RMAX, r = lane % RMAX;
      if (r < p.rows && j0 + c < p.N) gemv_store(p, out, r, j0 + c, v);
    } else {  // one row of x: the same products for every output row
      static_assert(RMAX == 1 && kCols <= 4, "one row");
#pragma unroll
      for (int c = 0; c < kCols; ++c)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
#pragma unroll
      for (int c = 0; c < kCols; ++c)
        if (lane < p.rows && j0 + c < p.N) gemv_store(p, out, lane, j0 + c, acc[c]);
    }
  }
}

// The same products for 2 to 8 rows and a large weight (the modulation of every active branch),
// with the weight streamed through shared memory: an item's 32 columns are one contiguous block
// of 64 K bytes, which a producer warp fetches whole (cp.async.bulk) into one of two buffers while
// the other 8 warps multiply the item before it, 4 columns each.  With direct loads a warp had
// only its own current columns in flight and stopped for every reduction: 56 x 3456 x 1152 took
// 168 us for 446 MB.
constexpr int kStreamCols = 32;
constexpr int kStreamThreads = 288;
inline size_t gemv_stream_smem(int K) {
  return static_cast<size_t>(8) * K * sizeof(float) + 2 * static_cast<size_t>(kStreamCols) * K * sizeof(bf16) + 64;
}

__global__ void __launch_bounds__(kStreamThreads, 1) gemv_stream_kernel(const GemvParams p, int* status) {
  extern __shared__ __align__(128) float xs[];  // x [8][2 planes][K / 2], two weight buffers, barriers
  const int K = p.K, half = K >> 1;
  uint8_t* wbuf = reinterpret_cast<uint8_t*>(xs + 8 * K);
  const uint32_t wbytes = kStreamCols * K * sizeof(bf16);
  uint64_t* full = reinterpret_cast<uint64_t*>(wbuf + 2 * wbytes);
  uint64_t* empty = full + 2;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 8);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  pdl_wait_and_trigger();
  const int k4 = K >> 2;
  for (int i = threadIdx.x; i < 8 * k4; i += kStreamThreads) {
    const int r = i / k4, k = (i - r * k4) << 2;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);  // rows past the last contribute nothing and are not stored
    if (r < p.rows) x = ld_f32x4(p.x + static_cast<int64_t>(r) * p.ldx + k);
    if (p.in_silu) x = make_float4(silu_f(x.x), silu_f(x.y), silu_f(x.z), silu_f(x.w));
    *reinterpret_cast<float4*>(xs + r * K + ((k & 4) ? half : 0) + (k >> 3) * 4) = x;
  }
  __syncthreads();
  const int per_seg = (p.N + kStreamCols - 1) / kStreamCols;
  const int n_items = per_seg * (p.n_seg > 0 ? p.n_seg : 1);
  if (warp == 8) {
    if (lane == 0) {
      int it = 0;
      for (int item = blockIdx.x; item < n_items; item += gridDim.x, ++it) {
        const int s = it & 1;
        if (!mbar_wait(&empty[s], ((it >> 1) & 1) ^ 1u, abort_flag, status, 41)) break;
        const int seg = item / per_seg, j0 = (item - seg * per_seg) * kStreamCols;
        const uint32_t bytes = min(kStreamCols, p.N - j0) * K * sizeof(bf16);  // K % 8 == 0: a multiple of 16
        mbar_arrive_expect_tx(&full[s], bytes);
        bulk_load(wbuf + s * wbytes, (p.n_seg ? p.w_seg[seg] : p.W) + static_cast<int64_t>(j0) * K, bytes, &full[s]);
      }
      if (*abort_flag)
        for (int i = it > 2 ? it - 2 : 0; i < it; ++i) mbar_drain(&full[i & 1], (i >> 1) & 1);
    }
    return;
  }
  int it = 0;
  for (int item = blockIdx.x; item < n_items; item += gridDim.x, ++it) {
    const int s = it & 1;
    const int seg = item / per_seg, j0 = (item - seg * per_seg) * kStreamCols;
    if (!mbar_wait_warp(smem_u32(&full[s]), (it >> 1) & 1, abort_flag, status, 42)) break;
    const uint8_t* W = wbuf + s * wbytes + static_cast<size_t>(warp) * 4 * K * sizeof(bf16);
    uint64_t acc2[32];  // [column][row], sums over even and odd k
#pragma unroll
    for (int i = 0; i < 32; ++i) acc2[i] = 0;
    // (columns past N hold whatever the buffer held; their sums are not stored)
    for (int k = lane * 8; k < K; k += 256) {
      uint64_t wf[4][4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint4 w = *reinterpret_cast<const uint4*>(W + (static_cast<size_t>(c) * K + k) * sizeof(bf16));
        const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) wf[c][q] = pack_f32x2(u[q] << 16, u[q] & 0xffff0000u);
      }
      const int xo = (k >> 3) * 4;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const ulonglong2 xa = *reinterpret_cast<const ulonglong2*>(xs + r * K + xo);
        const ulonglong2 xb = *reinterpret_cast<const ulonglong2*>(xs + r * K + half + xo);
        const uint64_t xv[4] = {xa.x, xa.y, xb.x, xb.y};
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc2[c * 8 + r] = fma_f32x2(wf[c][q], xv[q], acc2[c * 8 + r]);
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = sum_f32x2(acc2[i]);
    const float v = transpose_reduce32(acc, lane);
    const int j = j0 + warp * 4 + lane / 8, r = lane % 8;
    if (r < p.rows && j < p.N) gemv_store(p, p.n_seg ? p.out_seg[seg] : p.out, r, j, v);
  }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// A warp takes two rows: it normalises (and AdaLN modulates) them into its part of shared memory
// and multiplies them by 16 output channels' bf16 weight rows at a time, whose loads serve both
// rows (the weights come from L1: out_channels x K x 2 bytes per warp).  The 32 partial sums of a
// lane are reduced over the warp by one transpose reduction, after which lane l holds channel
// l / 2 of row l % 2.  One channel at a time, with its own reduction, was a chain of load and
// shuffle latencies (29 us for 2048 x 1152 and 16 channels), and with the rows in registers the
// unrolled code was as long as the work (26 us).
__global__ void __launch_bounds__(128, 3) head_small_kernel(const HeadParams p) {
  extern __shared__ float xh[];  // [warp][2][K]
  pdl_wait_and_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t r0 = (static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + warp) * 2;
  const int64_t rows = static_cast<int64_t>(p.batch) * p.n_tokens;
  if (r0 >= rows) return;
  const int nv = p.K >> 2;
  float4* x0 = reinterpret_cast<float4*>(xh + static_cast<size_t>(2 * warp) * p.K);
#pragma unroll 1
  for (int q = 0; q < 2; ++q) {
    const int64_t r = min(r0 + q, rows - 1);  // past the last row: computed again, not stored
    const int b = static_cast<int>(r / p.n_tokens);
    const float* x = p.h + r * p.ldx;
    float4* xs = x0 + q * nv;
    float s1 = 0.f, sq = 0.f;
#pragma unroll 4
    for (int i = lane; i < nv; i += 32) {
      const float4 v = ld_f32x4(x + 4 * i);
      xs[i] = v;
      s1 += (v.x + v.y) + (v.z + v.w);
    }
    const float mean = p.norm_kind != SGD_NORM_RMS ? warp_sum(s1) / p.K : 0.f;
#pragma unroll 4
    for (int i = lane; i < nv; i += 32) {
      const float4 v = xs[i];
      const float a0 = v.x - mean, a1 = v.y - mean, a2 = v.z - mean, a3 = v.w - mean;
      sq += (a0 * a0 + a1 * a1) + (a2 * a2 + a3 * a3);
    }
    const float rstd = rsqrtf(warp_sum(sq) / p.K + p.eps);
    const float* sh = p.shift ? p.shift + static_cast<int64_t>(b) * p.ld_mod : nullptr;
    const float* sc = p.scale ? p.scale + static_cast<int64_t>(b) * p.ld_mod : nullptr;
#pragma unroll 2
    for (int i = lane; i < nv; i += 32) xs[i] = norm_affine4(p, i, xs[i], mean, rstd, sc, sh);
  }
  // this lane's output row and channel within a group (each lane reads back what it wrote)
  const int64_t ro = r0 + (lane & 1);
  const int n = static_cast<int>(ro % p.n_tokens), b = static_cast<int>(ro / p.n_tokens);
  float* out = reinterpret_cast<float*>(p.slot->out) +
               (static_cast<int64_t>(b) * (p.n_tokens - p.n_prefix) + (n - p.n_prefix)) * p.out_channels;
  const bool store = ro < rows && n >= p.n_prefix;
#pragma unroll 1
  for (int c0 = 0; c0 < p.out_channels; c0 += 16) {
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.f;
#pragma unroll 2
    for (int i = lane; i < nv; i += 32) {
      uint2 w[16];  // channels past the last repeat it, not stored
#pragma unroll
      for (int c = 0; c < 16; ++c)
        w[c] = __ldg(reinterpret_cast<const uint2*>(p.W + static_cast<int64_t>(min(c0 + c, p.out_channels - 1)) * p.K) + i);
      const float4 u = x0[i], v = x0[nv + i];
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const float4 wf = bf16x4(w[c]);
        acc[2 * c] = fmaf(u.w, wf.w, fmaf(u.z, wf.z, fmaf(u.y, wf.y, fmaf(u.x, wf.x, acc[2 * c]))));
        acc[2 * c + 1] = fmaf(v.w, wf.w, fmaf(v.z, wf.z, fmaf(v.y, wf.y, fmaf(v.x, wf.x, acc[2 * c + 1]))));
      }
    }
    const float res = transpose_reduce32(acc, lane);
    const int c = c0 + (lane >> 1);
    if (store && c < p.out_channels) out[c] = res;
  }
}

__global__ void copy_out_kernel(const IoSlot* slot, const float* h, int64_t n4) {
  pdl_wait_and_trigger();
  float4* o = reinterpret_cast<float4*>(slot->out);
  const float4* s = reinterpret_cast<const float4*>(h);
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n4; i += stride)
    o[i] = s[i];
}

// Thread (x, y): 8 columns of every gridDim.y-th row (d % 8 == 0).
__global__ void __launch_bounds__(128) pack_f16_kernel(f16* dst, int ld_dst, int col0, const float* h, int rows, int d) {
  pdl_wait_and_trigger();
  const int c = (blockIdx.x * blockDim.x + threadIdx.x) * 8;
  if (c >= d) return;
  for (int r = blockIdx.y; r < rows; r += gridDim.y) {
    const float4* src = reinterpret_cast<const float4*>(h + static_cast<int64_t>(r) * d + c);
    const float4 a = src[0], b = src[1];
    const float f[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    *reinterpret_cast<uint4*>(dst + static_cast<int64_t>(r) * ld_dst + col0 + c) = pack_f16x8(f);
  }
}

// max |w| over a bf16 tensor: per-block maxima combined with an integer atomicMax on
// the float bit pattern (valid for non-negative floats); *out must start at 0.
__global__ void absmax_bf16_kernel(const bf16* w, int64_t n, float* out) {
  __shared__ float red[8];
  float m = 0.f;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride)
    m = fmaxf(m, fabsf(__bfloat162float(w[i])));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < (blockDim.x >> 5); ++i) m = fmaxf(m, red[i]);
    atomicMax(reinterpret_cast<int*>(out), __float_as_int(m));
  }
}

// dst = fp16(w * 2^shift): exact for every bf16 value whose scaled magnitude lies in
// the normal fp16 range (bf16 keeps 8 significant bits, fp16 11).
__global__ void convert_bf16_f16_kernel(const bf16* w, f16* dst, int64_t n, float scale) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride)
    dst[i] = __float2half_rn(sat_f16(__bfloat162float(w[i]) * scale));
}

// max |W[j, k] g[k]| (non-negative floats compared as integers, as absmax_bf16_kernel).
__global__ void absmax_scaled_kernel(const bf16* w, const bf16* g, int64_t n, int K, float* out) {
  __shared__ float red[8];
  float m = 0.f;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride)
    m = fmaxf(m, fabsf(__bfloat162float(w[i]) * __bfloat162float(g[i % K])));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < (blockDim.x >> 5); ++i) m = fmaxf(m, red[i]);
    atomicMax(reinterpret_cast<int*>(out), __float_as_int(m));
  }
}

// dst = fp16(W[j, k] g[k] 2^shift): the product of two bf16 values is exact in fp32, and
// is rounded once to fp16.
__global__ void convert_scaled_kernel(const bf16* w, const bf16* g, f16* dst, int64_t n, int K,
                                      float scale) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride)
    dst[i] = __float2half_rn(sat_f16(__bfloat162float(w[i]) * __bfloat162float(g[i % K]) * scale));
}

// One warp per row j: out[j] = scale sum_k W[j, k] (x[k] or 1), accumulated in double.
template <typename TW>
__global__ void rowdot_kernel(const TW* w, const bf16* x, int64_t rows, int K, float scale, float* out) {
  const int64_t j = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (j >= rows) return;
  double acc = 0.0;
  for (int k = lane; k < K; k += 32) {
    const double wv = static_cast<double>(static_cast<float>(w[j * K + k]));
    acc += x ? wv * static_cast<double>(__bfloat162float(x[k])) : wv;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) out[j] = static_cast<float>(acc * scale);
}

// z and eps 16-byte aligned: 4 elements per thread and step, the rest by the first threads
// (2.6 M elements: 8.1 us with one element per thread).
__global__ void sampler_kernel(float* z, const float* eps, float alpha, float beta, int64_t n, int vec) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  int64_t done = 0;
  if (vec) {
    const int64_t n4 = n >> 2;
    float4* z4 = reinterpret_cast<float4*>(z);
    const float4* e4 = reinterpret_cast<const float4*>(eps);
    for (int64_t i = i0; i < n4; i += stride) {
      float4 a = z4[i];
      const float4 e = e4[i];
      a.x = alpha * a.x - beta * e.x;
      a.y = alpha * a.y - beta * e.y;
      a.z = alpha * a.z - beta * e.z;
      a.w = alpha * a.w - beta * e.w;
      z4[i] = a;
    }
    done = n4 << 2;
  }
  for (int64_t i = done + i0; i < n; i += stride) z[i] = alpha * z[i] - beta * eps[i];
}

int grid_for(int64_t work, int threads) {
  const int64_t cap = static_cast<int64_t>(num_sms()) * 8;
  int64_t g = (work + threads - 1) / threads;
  if (g > cap) g = cap;
  return g < 1 ? 1 : static_cast<int>(g);
}

}  // namespace

namespace {
template <int MODE>
cudaError_t norm_launch_mode(const NormParams& p, cudaStream_t s) {
  const dim3 grid((p.rows + 3) / 4), block(128);
  if (p.d <= 256) return launch_k(norm_warp_kernel<2, MODE>, grid, block, 0, s, p);
  if (p.d <= 512) return launch_k(norm_warp_kernel<4, MODE>, grid, block, 0, s, p);
  if (p.d <= 1024) return launch_k(norm_warp_kernel<8, MODE>, grid, block, 0, s, p);
  if (p.d <= 1280) return launch_k(norm_warp_kernel<10, MODE>, grid, block, 0, s, p);
  if (p.d <= 2048) return launch_k(norm_warp_kernel<16, MODE>, grid, block, 0, s, p);
  if (p.rows <= wide_blocks(MODE, false) * num_sms())
    return launch_k(norm_wide_kernel<MODE, false>, dim3(p.rows), dim3(wide_threads(false)), 0, s, p);
  return launch_k(norm_wide_kernel<MODE, true>, dim3(wide_blocks(MODE, true) * num_sms()), dim3(wide_threads(true)), 0, s, p);
}
}  // namespace

cudaError_t norm_launch(const NormParams& p, cudaStream_t s) {
  if (!p.scale) return norm_launch_mode<kGain>(p, s);
  // the modulation may lie at any float's address
  const bool vec = p.ld_mod % 4 == 0 &&
                   ((reinterpret_cast<uintptr_t>(p.shift) | reinterpret_cast<uintptr_t>(p.scale)) & 15u) == 0;
  return vec && !p.g && !p.b ? norm_launch_mode<kMod>(p, s) : norm_launch_mode<kAny>(p, s);
}

cudaError_t wait_selftest_launch(int* status, int code, cudaStream_t s) {
  wait_selftest_kernel<<<1, 32, 0, s>>>(status, code);
  return cudaGetLastError();
}

cudaError_t drift_launch(const DriftParams& p, cudaStream_t s) {
  return launch_k(drift_kernel, dim3(kDriftBlocks), dim3(256), 0, s, p);
}

cudaError_t drift_reduce_launch(const float* partials, int n_groups, double* sums, cudaStream_t s) {
  return launch_k(drift_reduce_kernel, dim3(n_groups), dim3(32), 0, s, partials, sums);
}

cudaError_t frozen_launch(const FrozenParams& p, cudaStream_t s) {
  if (p.h16) {
    if (!p.stat || p.d % 8 || p.rows < 1 || frozen_stat_slots(p.d) > kStatSlots) return cudaErrorInvalidValue;
    const int64_t warps = static_cast<int64_t>(p.rows) * frozen_stat_slots(p.d);
    return launch_k(frozen_rows_kernel, dim3(static_cast<unsigned>((warps + 7) / 8)), dim3(256), 0, s, p);
  }
  return launch_k(frozen_kernel, dim3(grid_for(p.n / 8, 256)), dim3(256), 0, s, p);
}

cudaError_t io_set_launch(IoSlot* slot, const IoSlot& v, const TimeEmb& te, cudaStream_t s) {
  io_set_kernel<<<std::max(1, (te.n + 31) / 32), 32, 0, s>>>(slot, v, te);
  return cudaGetLastError();
}

cudaError_t stem_launch(const StemParams& p, cudaStream_t s) {
  const int rows = p.batch * p.n_tokens;
  if (p.kind != SGD_STEM_PATCH && p.kind != SGD_STEM_PATCH_TOKENS) {
    // about 16 blocks of 128 threads per SM, as far as there are rows (d % 8 == 0, checked at creation)
    const int gx = (p.d / 8 + 127) / 128;
    const int gy = std::max(1, std::min(rows, 16 * num_sms() / gx));
    return launch_k(stem_rows_kernel, dim3(gx, gy), dim3(128), 0, s, p);
  }
  const dim3 grid(((p.d / 4 + 127) / 128) * ((rows + kPatchRows - 1) / kPatchRows));
  if (p.d_in == 8) return launch_k(stem_patch_kernel<8>, grid, dim3(128), 0, s, p);
  if (p.d_in == 16) return launch_k(stem_patch_kernel<16>, grid, dim3(128), 0, s, p);
  if (p.d_in % 8 == 0) {
    const int64_t total4 = static_cast<int64_t>(rows) * (p.d / 4);
    return launch_k(stem_patch_any_kernel, dim3(static_cast<unsigned>((total4 + 255) / 256)), dim3(256), 0, s, p);
  }
  const int64_t total = static_cast<int64_t>(rows) * p.d;
  return launch_k(stem_kernel, dim3(static_cast<unsigned>((total + 255) / 256)), dim3(256), 0, s, p);
}

template <int RMAX, int COLS>
cudaError_t gemv_launch_r(const GemvParams& p, size_t smem, cudaStream_t s) {
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(gemv_kernel<RMAX, COLS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  const int cols_per_block = 8 * COLS;
  const int64_t items = static_cast<int64_t>((p.N + cols_per_block - 1) / cols_per_block) * (p.n_seg > 0 ? p.n_seg : 1);
  const int grid = static_cast<int>(std::min<int64_t>(items, 2 * static_cast<int64_t>(num_sms())));
  return launch_k(gemv_kernel<RMAX, COLS>, dim3(grid), dim3(256), smem, s, p);
}

cudaError_t gemv_launch(const GemvParams& p, cudaStream_t s) {
  const int xrows = p.ldx == 0 ? 1 : p.rows;
  const size_t smem = static_cast<size_t>(xrows) * p.K * sizeof(float);
  if (p.rows > 16 || smem > 200 * 1024 || (p.K % 8) || p.n_seg < 0 || p.n_seg > kGemvMaxSeg ||
      (p.n_seg > 0 && (p.out_silu || p.add_class || p.add_vec)) ||
      (p.ldx % 4) || (reinterpret_cast<uintptr_t>(p.x) & 15u))
    return cudaErrorInvalidValue;
  const bool few = static_cast<int64_t>(p.N) * std::max(p.n_seg, 1) < 32ll * num_sms();
  if (xrows == 1) {
    return few ? gemv_launch_r<1, 1>(p, smem, s) : gemv_launch_r<1, 4>(p, smem, s);
  }
  // many columns of a wide-enough weight to keep every SM streaming, and buffers that fit
  const int64_t items = static_cast<int64_t>((p.N + kStreamCols - 1) / kStreamCols) * std::max(p.n_seg, 1);
  if (xrows <= 8 && items >= 2 * num_sms() && gemv_stream_smem(p.K) <= 220 * 1024) {
    const size_t bytes = gemv_stream_smem(p.K);
    cudaError_t e = cudaFuncSetAttribute(gemv_stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(bytes));
    if (e != cudaSuccess) return e;
    return launch_k(gemv_stream_kernel, dim3(num_sms()), dim3(kStreamThreads), bytes, s, p, device_status_ptr());
  }
  if (xrows <= 8) return few ? gemv_launch_r<8, 1>(p, smem, s) : gemv_launch_r<8, 4>(p, smem, s);
  return gemv_launch_r<16, 2>(p, smem, s);
}

cudaError_t head_small_launch(const HeadParams& p, cudaStream_t s) {
  const int64_t rows = static_cast<int64_t>(p.batch) * p.n_tokens;
  if (p.K % 4 || p.K > 4096 || p.out_channels > 64 || p.out_channels > p.N || p.ldx % 4 ||
      (p.shift && p.ld_mod % 4))
    return cudaErrorInvalidValue;
  const size_t smem = static_cast<size_t>(8) * p.K * sizeof(float);  // 4 warps of 2 rows: 128 KB at most
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(head_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  return launch_k(head_small_kernel, dim3(static_cast<unsigned>((rows + 7) / 8)), dim3(128), smem, s, p);
}

cudaError_t copy_out_launch(const IoSlot* slot, const float* h, int64_t n, cudaStream_t s) {
  return launch_k(copy_out_kernel, dim3(grid_for(n / 4, 256)), dim3(256), 0, s, slot, h, n / 4);
}

cudaError_t pack_f16_launch(f16* dst, int ld_dst, int col0, const float* h, int rows, int d,
                            cudaStream_t s) {
  const int gx = (d / 8 + 127) / 128;
  return launch_k(pack_f16_kernel, dim3(gx, std::max(1, std::min(rows, 16 * num_sms() / gx))), dim3(128), 0, s, dst,
                  ld_dst, col0, h, rows, d);
}

cudaError_t absmax_bf16_launch(const bf16* w, int64_t n, float* out, cudaStream_t s) {
  absmax_bf16_kernel<<<grid_for(n, 256), 256, 0, s>>>(w, n, out);
  return cudaGetLastError();
}

cudaError_t convert_bf16_f16_launch(const bf16* w, f16* dst, int64_t n, int shift, cudaStream_t s) {
  convert_bf16_f16_kernel<<<grid_for(n, 256), 256, 0, s>>>(w, dst, n, ldexpf(1.0f, shift));
  return cudaGetLastError();
}

cudaError_t absmax_scaled_launch(const bf16* w, const bf16* g, int64_t rows, int K, float* out,
                                 cudaStream_t s) {
  absmax_scaled_kernel<<<grid_for(rows * K, 256), 256, 0, s>>>(w, g, rows * K, K, out);
  return cudaGetLastError();
}

cudaError_t convert_scaled_launch(const bf16* w, const bf16* g, f16* dst, int64_t rows, int K, int shift,
                                  cudaStream_t s) {
  convert_scaled_kernel<<<grid_for(rows * K, 256), 256, 0, s>>>(w, g, dst, rows * K, K, ldexpf(1.0f, shift));
  return cudaGetLastError();
}

cudaError_t rowsum_f16_launch(const f16* w, int64_t rows, int K, float scale, float* out, cudaStream_t s) {
  rowdot_kernel<f16><<<static_cast<unsigned>((rows + 7) / 8), 256, 0, s>>>(w, nullptr, rows, K, scale, out);
  return cudaGetLastError();
}

cudaError_t rowdot_bf16_launch(const bf16* w, const bf16* x, int64_t rows, int K, float* out,
                               cudaStream_t s) {
  rowdot_kernel<bf16><<<static_cast<unsigned>((rows + 7) / 8), 256, 0, s>>>(w, x, rows, K, 1.f, out);
  return cudaGetLastError();
}

cudaError_t sampler_launch(float* z, const float* eps, float alpha, float beta, int64_t n,
                           cudaStream_t s) {
  const int vec = ((reinterpret_cast<uintptr_t>(z) | reinterpret_cast<uintptr_t>(eps)) & 15u) == 0 ? 1 : 0;
  sampler_kernel<<<grid_for(vec ? (n + 3) / 4 : n, 256), 256, 0, s>>>(z, eps, alpha, beta, n, vec);
  return cudaGetLastError();
}

}  // namespace sgd
