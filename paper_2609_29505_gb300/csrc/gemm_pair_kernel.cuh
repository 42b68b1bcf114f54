// The tcgen05 GEMM on CTA pairs (cta_group::2), C = A B^T with fused epilogues: the default
// kernel of every projection with more than one 128-row block.
//
// A cluster of two CTAs computes one 256 x BN output tile.  Each CTA loads its own 128 rows of
// A and half of B's BN rows per 64-wide K-block (16 KB + BN * 64 bytes), and the leader's
// tcgen05.mma (M = 256) reads both CTAs' shared memory and accumulates 128 rows in each CTA's
// TMEM.  A 1-CTA tile of 128 x 256 needs 48 KB per K-block for 512 tensor-core clocks, above
// the ~70 bytes per clock that reach an SM from L2 when all of them load; the pair needs 32 KB.
//
//   warp 0      TMA producer (both CTAs): its A rows and its half of B into a ring of stages.
//               Bytes of both CTAs are credited to the leader's `full` barrier.
//   warp 1      allocates TMEM (both CTAs); in the leader issues the MMAs, and commits every
//               stage's release and every finished accumulator to both CTAs.
//   warps 2-9   epilogue (both CTAs, each on its own 128 rows): warps w and w + 4 share TMEM
//               lanes 32 (w % 4) and split the columns.  Two accumulators, so that a tile's
//               epilogue overlaps the next tile's MMAs.
//
// Every wait is bounded as in the 1-CTA kernel; the cluster barriers (start, end) are reached
// by every thread because all other waits are.
#pragma once

#include "gemm_kernel.cuh"

namespace sgd {
namespace gk {

enum { kEpPlain = 0, kEpDelta = 1, kEpGated = 2, kEpRope = 3 };

template <int BN>
struct PairCfg {
  static constexpr int kBK = 64;
  static constexpr int kEpiWarps = 8;
  static constexpr int kThreads = 64 + 32 * kEpiWarps;
  static constexpr int kTmemCols = 2 * BN > 256 ? 512 : 256;
  static constexpr int kRowsB = BN / 2;
  static constexpr int kTileA = kBM * kBK * 2;
  static constexpr int kTileB = kRowsB * kBK * 2;
  static constexpr int kStageBytes = kTileA + kTileB;
  static constexpr int kStaging = kEpiWarps * 4096;
  static constexpr int kStages = (232448 - 1024 - 512 - kStaging) / kStageBytes;
  static constexpr int kSmemBytes = kStages * kStageBytes + kStaging + 1024 /*align*/ + 512 /*barriers*/;
  static_assert(BN % 32 == 0 && BN >= 64 && BN <= 256, "M = 256 instructions take N in steps of 32");
  static_assert(kTileB % 1024 == 0, "operand tiles start on 1024-byte boundaries");
  static_assert((2 * kStages + 5) * 8 + 4 * 4 <= 512, "barrier block");
};

// RoPE through the staging buffer: 16 columns of a head's first half and the 16 they rotate
// with go through shared memory together, and each lane rotates 4 pairs of a row, with cos and
// sin read 64 bytes per row.
template <class Src>
__device__ __forceinline__ void rope_staged(const TcArgs& a, void* out, int row, int n0, const Src& src, int cb,
                                            int ce, float4* stg) {
  const EpiParams& e = a.epi;
  const int lane = threadIdx.x & 31;
  const int row0 = row - lane;
  const int lr = lane >> 2, lc = lane & 3;
  const int dh = e.d_head, hd = dh >> 1;
  f16* o = reinterpret_cast<f16*>(out);
#pragma unroll 1
  for (int hb = cb; hb < ce; hb += dh) {
    if (n0 + hb >= a.N) break;  // N is a multiple of d_head or the head's columns are checked below
    const bool rot = n0 + hb < e.rope_cols;
#pragma unroll 1
    for (int j = 0; j < hd; j += 16) {
      float4 cs[4], sn[4];
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        cs[it] = make_float4(1.f, 1.f, 1.f, 1.f);
        sn[it] = make_float4(0.f, 0.f, 0.f, 0.f);
        const int r = row0 + it * 8 + lr;
        if (rot && r < a.M) {
          const int64_t at = static_cast<int64_t>(r % e.rope_tokens) * hd + j + 4 * lc;
          cs[it] = *reinterpret_cast<const float4*>(e.rope_cos + at);
          sn[it] = *reinterpret_cast<const float4*>(e.rope_sin + at);
        }
      }
      {
        float x[16], y[16];
        src.load2(hb + j, hb + hd + j, x, y);
        stage_put16_f32(stg, 0, x);
        stage_put16_f32(stg, 1, y);
      }
      __syncwarp();
      const int c1 = n0 + hb + j + 4 * lc, c2 = c1 + hd;
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        const int r = it * 8 + lr;
        const float4 p = stg[r * 8 + (lc ^ (r & 7))], q = stg[r * 8 + ((lc + 4) ^ (r & 7))];
        float4 u = p, v = q;
        if (rot) {
          const float4 c = cs[it], s = sn[it];
          u = make_float4(p.x * c.x - q.x * s.x, p.y * c.y - q.y * s.y, p.z * c.z - q.z * s.z, p.w * c.w - q.w * s.w);
          v = make_float4(q.x * c.x + p.x * s.x, q.y * c.y + p.y * s.y, q.z * c.z + p.z * s.z, q.w * c.w + p.w * s.w);
        }
        if (row0 + r < a.M) {
          f16* orow = o + static_cast<int64_t>(row0 + r) * e.ldo;
          if (c1 < a.N) *reinterpret_cast<uint2*>(orow + c1) = pack_f16x4(u);
          if (c2 < a.N) *reinterpret_cast<uint2*>(orow + c2) = pack_f16x4(v);
        }
      }
      __syncwarp();  // the next chunk overwrites the staging buffer
    }
  }
}

template <int BN, int EP, class Src>
__device__ __forceinline__ void pair_epilogue(const TcArgs& a, void* out, int row, int n_blk, const Src& src,
                                              int part, float4* stg, float4* hv) {
  const EpiParams& e = a.epi;
  const int row0 = row - (threadIdx.x & 31);
  if constexpr (EP == kEpDelta) {
    constexpr int kSplit = ((BN / 32 + 1) / 2) * 32;
    delta_staged<std::is_same<Src, TmemSrc>::value>(a, row, n_blk * BN, src, part ? kSplit : 0, part ? BN : kSplit,
                                                    stg, hv);
  } else if constexpr (EP == kEpRope) {
    rope_staged(a, out, row, n_blk * BN, src, part ? BN / 2 : 0, part ? BN : BN / 2, stg);
  } else if constexpr (EP == kEpGated) {
    constexpr int kOut = BN / 2, kSplit = ((kOut / 32 + 1) / 2) * 32;
    const int n0 = n_blk * kOut, ce = part ? kOut : kSplit;
#pragma unroll 1
    for (int c = part ? kSplit : 0; c < ce; c += 32) {
      if (n0 + c >= a.N) break;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int cc = c + 16 * half;
        if (kOut % 32 != 0 && cc >= kOut) break;
        float x[16], y[16];
        src.load2(cc, kOut + cc, x, y);
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = e.act ? x[i] * gelu_erf_f(y[i]) : silu_f(x[i]) * y[i];
        stage_put16_f16(stg, half, x);
      }
      stage_flush_f16(e, out, row0, a.M, min(a.N, n0 + kOut), n0 + c, stg);
    }
  } else {
    constexpr int kSplit = ((BN / 32 + 1) / 2) * 32;
    const int n0 = n_blk * BN, ce = part ? BN : kSplit;
#pragma unroll 1
    for (int c = part ? kSplit : 0; c < ce; c += 32) {
      if (n0 + c >= a.N) break;
      float x[16], y[16];
      src.load2(c, c + 16, x, y);
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        float* v = half ? y : x;
        if (e.kind == SGD_EPI_GELU) {
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = e.act ? gelu_erf_f(v[i]) : gelu_tanh_f(v[i]);
        }
        if (e.kind == SGD_EPI_F32)
          stage_put16_f32(stg, half, v);
        else
          stage_put16_f16(stg, half, v);
      }
      if (e.kind == SGD_EPI_F32)
        stage_flush_f32(e, out, row0, a.M, a.N, n0 + c, stg);
      else
        stage_flush_f16(e, out, row0, a.M, a.N, n0 + c, stg);
    }
  }
}

// Work is dealt out to pairs as the 1-CTA kernel deals it to CTAs (CtaWork; stream-K segments
// first).  A stream-K tile has one workspace slot and one ticket per CTA of the pair: each
// CTA's 128 rows are summed and finished on their own.
template <int BN, int EP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PairCfg<BN>::kThreads, 1)
    gemm_pair_kernel(const __grid_constant__ TcArgs a) {
  using C = PairCfg<BN>;
  constexpr int kStages = C::kStages, kTileA = C::kTileA, kStageBytes = C::kStageBytes;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(tiles + kStages * kStageBytes);
  uint64_t* empty = full + kStages;
  uint64_t* tfull = empty + kStages;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* last_flag = reinterpret_cast<volatile int*>(tmem_slot + 2);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 2 * C::kEpiWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&a.tmap_a);
    tma_prefetch_desc(&a.tmap_b);
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, C::kTmemCols);
  tc_fence_before();
  __syncthreads();
  __syncwarp();
  cluster_sync();
  tc_fence_after();
  pdl_wait_and_trigger();  // the prologue above touched only shared memory and TMEM
  const uint32_t tmem_base = *tmem_slot;
  const CtaWork w = cta_work(a, a.num_m * a.num_n, pair, num_pairs, pair);

  if (warp == 0) {
    const bool lead = elect_one();
    const uint32_t tiles0 = smem_u32(tiles), empty0 = smem_u32(empty);
    const uint32_t full0 = map_to_rank(smem_u32(full), 0);  // the leader's barriers
    uint32_t st = 0, ph = 1;
    int it = 0;
    bool ok = true;
    for (int u = 0; u < w.n_units && ok; ++u) {
      int tile, k0, k1;
      unit_at(a, w, u, tile, k0, k1);
      int m_blk, n_blk;
      tile_coords(a, tile, m_blk, n_blk);
      const int row_a = (2 * m_blk + static_cast<int>(rank)) * kBM;
      // gated: the leader's half of B is the gate rows, the other CTA's the up rows
      const int row_b = EP == kEpGated ? static_cast<int>(rank) * a.N + n_blk * C::kRowsB
                                       : n_blk * BN + static_cast<int>(rank) * C::kRowsB;
      for (int kb = k0; kb < k1; ++kb, ++it) {
        if (!mbar_wait_warp(empty0 + 8 * st, ph, abort_flag, a.status, 31)) {
          ok = false;
          break;
        }
        if (lead) {
          const uint32_t bar = full0 + 8 * st, dst = tiles0 + st * kStageBytes;
          if (rank == 0) mbar_arrive_expect_tx_at(smem_u32(full) + 8 * st, 2 * kStageBytes);
          tma_load_2d_pair(dst, &a.tmap_a, bar, kb * C::kBK, row_a);
          tma_load_2d_pair(dst + kTileA, &a.tmap_b, bar, kb * C::kBK, row_b);
        }
        if (++st == kStages) {
          st = 0;
          ph ^= 1;
        }
      }
    }
    const int tail = it > kStages ? it - kStages : 0;  // the latest issue of each stage
    if (*abort_flag) {
      // both CTAs' loads still in flight; the other CTA stays at the cluster barrier meanwhile
      if (lead && rank == 0)
        for (int i = tail; i < it; ++i) drain_wait(&full[i % kStages], (i / kStages) & 1);
    } else if (lead) {
      // the releases committed to this CTA's barriers arrive before it ends
      for (int i = tail; i < it; ++i) drain_wait(&empty[i % kStages], (i / kStages) & 1);
    }
  } else if (warp == 1) {
    if (rank == 0) {
      const bool lead = elect_one();
      constexpr uint32_t idesc = umma_idesc_f16(2 * kBM, BN);
      const uint32_t full0 = smem_u32(full), empty0 = smem_u32(empty);
      const uint64_t desc_a0 = smem_desc_sw128(smem_u32(tiles)), desc_b0 = smem_desc_sw128(smem_u32(tiles) + kTileA);
      uint64_t da = desc_a0, db = desc_b0;
      uint32_t st = 0, ph = 0;
      bool ok = true, ready = false;
      for (int u = 0; u < w.n_units && ok; ++u) {
        int tile, k0, k1;
        unit_at(a, w, u, tile, k0, k1);
        const int acc = u & 1;
        const uint32_t aph = (u >> 1) & 1;
        if (!mbar_wait_warp(smem_u32(&tempty[acc]), aph ^ 1u, abort_flag, a.status, 32)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * BN;
        uint32_t accumulate = 0;
        for (int kb = k0; kb < k1; ++kb) {
          if (!ready && !mbar_wait_warp(full0 + 8 * st, ph, abort_flag, a.status, 33)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t bar = empty0 + 8 * st;
          if (lead) {
            umma_f16_pair(d_tmem, da, db, idesc, accumulate);
            umma_f16_pair(d_tmem, da + 2, db + 2, idesc, 1u);
          }
          accumulate = 1;
          const uint64_t ca = da, cb = db;
          da += kStageBytes >> 4;
          db += kStageBytes >> 4;
          if (++st == kStages) {
            st = 0;
            ph ^= 1;
            da = desc_a0;
            db = desc_b0;
          }
          ready = mbar_test_warp(full0 + 8 * st, ph);
          if (lead) {
            umma_f16_pair(d_tmem, ca + 4, cb + 4, idesc, 1u);
            umma_f16_pair(d_tmem, ca + 6, cb + 6, idesc, 1u);
            umma_commit_pair(bar);
          }
        }
        if (!ok) break;
        if (lead) umma_commit_pair(smem_u32(&tfull[acc]));
      }
      if (lead) umma_commit_pair(smem_u32(drain));
    }
    // every MMA has finished, and the leader has committed for the last time, once `drain` completes
    if (lane == 0) drain_wait(drain, 0);
  } else {
    constexpr int kEpiThreads = 32 * C::kEpiWarps;
    float4* stg = reinterpret_cast<float4*>(tiles + kStages * kStageBytes + 512) + (warp - 2) * 256;
    const int q = warp & 3, part = (warp - 2) >> 2;
    constexpr int kSplit = ((BN / 32 + 1) / 2) * 32;
    const uint32_t tempty0 = map_to_rank(smem_u32(tempty), 0);
    const int total = a.sk_tiles * a.num_k;
    void* out = a.epi.out_slot ? *a.epi.out_slot : a.epi.out;
    float4 hv[8];  // first 32-column chunk of h (delta_staged)
    for (int u = 0; u < w.n_units; ++u) {
      int tile, k0, k1;
      unit_at(a, w, u, tile, k0, k1);
      int m_blk, n_blk;
      tile_coords(a, tile, m_blk, n_blk);
      const int acc = u & 1;
      const uint32_t aph = (u >> 1) & 1;
      const int row = (2 * m_blk + static_cast<int>(rank)) * kBM + q * 32 + lane;
      const uint32_t tbase = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + acc * BN;
      const bool whole = k0 == 0 && k1 == a.num_k;
      if (EP == kEpDelta && whole) {
        prefetch_h_row(a.epi, row, a.M, a.N, n_blk * BN, part ? kSplit : 0, part ? BN : kSplit);
        load_h_chunk(a, row - lane, n_blk * BN + (part ? kSplit : 0), hv);
      }
      const bool ok = mbar_wait_warp(smem_u32(&tfull[acc]), aph, abort_flag, a.status, 34);
      if (u >= w.n_sk || whole) {
        if (ok) {
          tc_fence_after();
          pair_epilogue<BN, EP>(a, out, row, n_blk, TmemSrc{tbase, a.epi.alpha}, part, stg, hv);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(tempty0 + 8 * acc);
        }
        if (u >= w.n_sk) {
          if (!ok) break;
        } else if (!epi_bar_and(ok, kEpiThreads)) {  // stream-K units are left together
          break;
        }
        continue;
      }
      // a part of the tile's K range: store it, draw a ticket; the last CTA sums and finishes
      const int first = sk_owner(tile * a.num_k, total, a.sk_ctas);
      const int nseg = sk_owner(tile * a.num_k + a.num_k - 1, total, a.sk_ctas) - first + 1;
      const int slot_tile = 2 * tile + static_cast<int>(rank);
      float* slot0 = a.ws + static_cast<size_t>(slot_tile) * a.max_seg * (kBM * BN);
      if (ok) {
        tc_fence_after();
        store_partial<BN>(slot0 + static_cast<size_t>(pair - first) * (kBM * BN), q * 32 + lane, tbase,
                          part ? kSplit : 0, part ? BN : kSplit);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(tempty0 + 8 * acc);
        __threadfence();
      }
      if (!epi_bar_and(ok, kEpiThreads)) break;
      if (threadIdx.x == 64) {
        __threadfence();
        *last_flag = atomicAdd(&a.sk_cnt[slot_tile], 1) == nseg - 1 ? 1 : 0;
      }
      epi_bar(kEpiThreads);
      if (*last_flag != 0) {
        __threadfence();
        pair_epilogue<BN, EP>(a, out, row, n_blk, WsSrc<BN>{slot0, nseg, q * 32 + lane, a.epi.alpha}, part, stg, hv);
        if (threadIdx.x == 64) a.sk_cnt[slot_tile] = 0;
      }
    }
  }

  tc_fence_before();
  __syncwarp();
  cluster_sync();  // nothing of either CTA refers to the other's memory any more
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem_base, C::kTmemCols);
}

template <int BN, int EP>
cudaError_t launch_pair(const GemmPlan& p, const TcArgs& a, cudaStream_t s) {
  using C = PairCfg<BN>;
  static bool attr_done[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr_done[dev]) {
    cudaError_t err = cudaFuncSetAttribute(gemm_pair_kernel<BN, EP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           C::kSmemBytes);
    if (err != cudaSuccess) return err;
    attr_done[dev] = true;
  }
  return launch_k(gemm_pair_kernel<BN, EP>, dim3(p.grid), dim3(C::kThreads), C::kSmemBytes, s, a);
}

}  // namespace gk
}  // namespace sgd
