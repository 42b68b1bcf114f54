// The tcgen05 GEMM C = A B^T with fused epilogues on CTA groups of one or two (CG), one
// instantiation per group, tile width and epilogue: the default kernel of every projection.
//
// CG = 2: a cluster of two CTAs computes one 256 x BN output tile (tcgen05 cta_group::2).  Each CTA
// loads its own 128 rows of A and half of B's BN rows per 64-wide K-block (16 KB + BN * 64 bytes),
// and the leader's tcgen05.mma (M = 256) reads both CTAs' shared memory and accumulates 128 rows
// in each CTA's TMEM.  A 1-CTA tile of 128 x 256 puts 48 KB per K-block into shared memory and
// reads them back in 512 tensor-core clocks, more than shared memory moves (it takes 692); the
// pair puts 32 KB there (528).  CG = 1: a CTA computes a 128 x BN tile by itself, for problems of few rows.
// One epilogue per instantiation keeps every value of it in registers (the kernel that holds
// all of them in one body spills) and the code that a short launch has to fetch small.
//
//   warp 0      TMA producer (every CTA): its A rows and its part of B into a ring of stages.
//               Bytes of a pair are credited to the leader's `full` barrier.
//   warp 1      allocates TMEM (every CTA); in the leader issues the MMAs, and commits every
//               stage's release and every finished accumulator to all CTAs of the group.
//   warps 2-9   epilogue (every CTA, on its own 128 rows): warps w and w + 4 share TMEM
//               lanes 32 (w % 4) and split the columns.  Two accumulators, so that a tile's
//               epilogue overlaps the next tile's MMAs.
//
// Every wait is bounded as in the kernel of gemm_kernel.cuh; the cluster barriers (start, end) are
// reached by every thread because all other waits are.
#pragma once

#include "gemm_kernel.cuh"

namespace sgd {
namespace gk {

enum { kEpPlain = 0, kEpDelta = 1, kEpGated = 2, kEpRope = 3 };

template <int CG, int BN>
struct GroupCfg {
  static constexpr int kBK = 64;
  static constexpr int kEpiWarps = 8;
  static constexpr int kThreads = 64 + 32 * kEpiWarps;
  static constexpr int kTmemCols = 2 * BN > 256 ? 512 : (2 * BN > 128 ? 256 : 128);
  static constexpr int kRowsB = BN / CG;
  static constexpr int kTileA = kBM * kBK * 2;
  static constexpr int kTileB = kRowsB * kBK * 2;
  static constexpr int kStageBytes = kTileA + kTileB;
  static constexpr int kStaging = kEpiWarps * 4096;
  static constexpr int kStages = (232448 - 1024 - 512 - kStaging) / kStageBytes;
  static constexpr int kSmemBytes = kStages * kStageBytes + kStaging + 1024 /*align*/ + 512 /*barriers*/;
  static_assert(CG == 1 || CG == 2, "one CTA or a pair");
  static_assert(BN % 32 == 0 && BN >= 64 && BN <= 256, "M = 256 instructions take N in steps of 32");
  static_assert(kTileB % 1024 == 0, "operand tiles start on 1024-byte boundaries");
  static_assert((2 * kStages + 5) * 8 + 4 * 4 <= 512, "barrier block");
};

// cos and sin of 4 pairs of each of a lane's 4 rows, and where the rows' tables start (-1: no row).
struct RopeTab {
  int64_t at[4];
  float4 cs[4], sn[4];
};
__device__ __forceinline__ void rope_load(const EpiParams& e, bool rot, int j, RopeTab& t) {
#pragma unroll
  for (int it = 0; it < 4; ++it) {
    if (rot && t.at[it] >= 0) {
      t.cs[it] = *reinterpret_cast<const float4*>(e.rope_cos + t.at[it] + j);
      t.sn[it] = *reinterpret_cast<const float4*>(e.rope_sin + t.at[it] + j);
    }
  }
}

// Column range cb .. ce and pairs j0 .. j1 of every head that a warp's half of a tile covers: whole
// heads, or half of the pairs of the tile's one head.
template <int BN>
struct RopeRange {
  int cb, ce, j0, j1;
  __device__ __forceinline__ RopeRange(int hd, int part) {
    const bool heads = 2 * hd <= BN / 2;
    cb = heads && part ? BN / 2 : 0;
    ce = heads && !part ? BN / 2 : BN;
    j0 = !heads && part ? hd / 2 : 0;
    j1 = !heads && !part ? hd / 2 : hd;
  }
};

// The tables of the first chunk, which the accumulator is not needed for.
template <int BN>
__device__ __forceinline__ void rope_begin(const TcArgs& a, int row0, int n0, int part, RopeTab& t) {
  const int lane = threadIdx.x & 31, hd = a.epi.d_head >> 1;
#pragma unroll
  for (int it = 0; it < 4; ++it) {
    const int r = row0 + it * 8 + (lane >> 2);
    t.at[it] = r < a.M ? static_cast<int64_t>(r % a.epi.rope_tokens) * hd + 4 * (lane & 3) : -1;
  }
  const RopeRange<BN> g(hd, part);
  rope_load(a.epi, n0 + g.cb < a.epi.rope_cols, g.j0, t);
}

// RoPE through the staging buffer: 16 columns of a head's first half and the 16 they rotate
// with go through shared memory together, and each lane rotates 4 pairs of a row, with cos and
// sin read 64 bytes per row.  The first chunk's tables are fetched before the accumulator is there
// and the next chunk's while one is rotated (read when a chunk needed them, each of a warp's 4
// chunks waited for L2: 64 x 768 x 256 6.65 -> 5.80 us, 333 x 12288 x 256 10.8 -> 9.9,
// 333 x 12288 x 4096 34.1 -> 32.9).
template <int BN, class Src>
__device__ __forceinline__ void rope_staged(const TcArgs& a, void* out, int row, int n0, const Src& src, int part,
                                            float4* stg, RopeTab& t) {
  const EpiParams& e = a.epi;
  const int lane = threadIdx.x & 31;
  const int row0 = row - lane;
  const int lr = lane >> 2, lc = lane & 3;
  const int dh = e.d_head, hd = dh >> 1;
  const RopeRange<BN> g(hd, part);
  f16* o = reinterpret_cast<f16*>(out);
#pragma unroll 1
  for (int hb = g.cb; hb < g.ce; hb += dh) {
    if (n0 + hb >= a.N) break;  // N is a multiple of d_head or the head's columns are checked below
    const bool rot = n0 + hb < e.rope_cols;
#pragma unroll 1
    for (int j = g.j0; j < g.j1; j += 16) {
      {
        float x[16], y[16];
        src.load2(hb + j, hb + hd + j, x, y);
        stage_put16_f32(stg, 0, x);
        stage_put16_f32(stg, 1, y);
      }
      __syncwarp();
      const RopeTab c = t;
      if (j + 16 < g.j1)
        rope_load(e, rot, j + 16, t);
      else if (hb + dh < g.ce)
        rope_load(e, n0 + hb + dh < e.rope_cols, g.j0, t);
      const int c1 = n0 + hb + j + 4 * lc, c2 = c1 + hd;
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        const int r = it * 8 + lr;
        const float4 p = stg[r * 8 + (lc ^ (r & 7))], q = stg[r * 8 + ((lc + 4) ^ (r & 7))];
        float4 u = p, v = q;
        if (rot) {
          const float4 cs = c.cs[it], s = c.sn[it];
          u = make_float4(p.x * cs.x - q.x * s.x, p.y * cs.y - q.y * s.y, p.z * cs.z - q.z * s.z, p.w * cs.w - q.w * s.w);
          v = make_float4(q.x * cs.x + p.x * s.x, q.y * cs.y + p.y * s.y, q.z * cs.z + p.z * s.z, q.w * cs.w + p.w * s.w);
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

template <int CG>
__device__ __forceinline__ void umma_group(uint32_t d, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
  if constexpr (CG == 2)
    umma_f16_pair(d, a_desc, b_desc, idesc, acc);
  else
    umma_f16(d, a_desc, b_desc, idesc, acc);
}
template <int CG>
__device__ __forceinline__ void umma_commit_group(uint32_t bar) {
  if constexpr (CG == 2)
    umma_commit_pair(bar);
  else
    umma_commit_at(bar);
}
template <int CG>
__device__ __forceinline__ void arrive_leader(uint32_t bar) {
  if constexpr (CG == 2)
    mbar_arrive_cluster(bar);
  else
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

template <int BN, int EP, class Src>
__device__ __forceinline__ void group_epilogue(const TcArgs& a, void* out, int row, int n_blk, const Src& src,
                                              int part, float4* stg, float4* hv, RopeTab& rt) {
  const EpiParams& e = a.epi;
  const int row0 = row - (threadIdx.x & 31);
  if constexpr (EP == kEpDelta) {
    constexpr int kSplit = ((BN / 32 + 1) / 2) * 32;
    delta_staged<true>(a, row, n_blk * BN, src, part ? kSplit : 0, part ? BN : kSplit,
                                                    stg, hv);
  } else if constexpr (EP == kEpRope) {
    rope_staged<BN>(a, out, row, n_blk * BN, src, part, stg, rt);
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
        if (e.act) {
#pragma unroll
          for (int i = 0; i < 16; ++i) x[i] *= gelu_erf_f(y[i]);
        } else {
#pragma unroll
          for (int i = 0; i < 16; i += 2) silu2(x[i], x[i + 1]);
#pragma unroll
          for (int i = 0; i < 16; ++i) x[i] *= y[i];
        }
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
        if (e.kind == SGD_EPI_GELU && e.act) {
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = gelu_erf_f(v[i]);
        } else if (e.kind == SGD_EPI_GELU) {
#pragma unroll
          for (int i = 0; i < 16; i += 2) gelu_tanh2(v[i], v[i + 1]);
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

// Persistent: group g computes tiles g, g + num_groups, ... over their whole K range.  (Splitting
// the K range of the tiles of a short last wave over all groups, through partial tiles in a
// workspace as in gemm_kernel.cuh, cost 9 to 20 us a launch and gained only at 64 x 4096 x 12288:
// 36.2 -> 32.6 us.)
template <int CG, int BN, int EP>
__device__ __forceinline__ void gemm_group_body(const TcArgs& a) {
  using C = GroupCfg<CG, BN>;
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

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = CG == 2 ? cluster_rank() : 0;
  const int group = blockIdx.x / CG, num_groups = gridDim.x / CG;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&a.tmap_a);
    tma_prefetch_desc(&a.tmap_b);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], CG * C::kEpiWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    if constexpr (CG == 2) {
      tmem_alloc_pair(tmem_slot, C::kTmemCols);
    } else {
      tmem_alloc(tmem_slot, C::kTmemCols);
      tmem_relinquish();
    }
  }
  const int num_tiles = a.num_m * a.num_n;
  tc_fence_before();
  __syncthreads();
  if constexpr (CG == 2) {
    __syncwarp();
    cluster_sync();
  }
  tc_fence_after();
  // B's part of a K-block into stage st, with the stage's expected bytes (A's too).  gated: half of
  // B's rows are the gate's, the other half the up projection's (of a pair, the leader's half and
  // the other CTA's)
  const auto load_b = [&](int n_blk, int kb, uint32_t st) {
    const uint32_t dst = smem_u32(tiles) + st * kStageBytes + kTileA;
    if constexpr (CG == 2) {
      const uint32_t bar = map_to_rank(smem_u32(full), 0) + 8 * st;  // the leader's barrier
      const int row_b = EP == kEpGated ? static_cast<int>(rank) * a.N + n_blk * C::kRowsB
                                       : n_blk * BN + static_cast<int>(rank) * C::kRowsB;
      if (rank == 0) mbar_arrive_expect_tx_at(smem_u32(full) + 8 * st, 2 * kStageBytes);
      tma_load_2d_pair(dst, &a.tmap_b, bar, kb * C::kBK, row_b);
    } else {
      const uint32_t bar = smem_u32(full) + 8 * st;
      mbar_arrive_expect_tx_at(bar, kStageBytes);
      tma_load_2d_at(dst, &a.tmap_b, bar, kb * C::kBK, EP == kEpGated ? n_blk * (BN / 2) : n_blk * BN);
      if (EP == kEpGated)
        tma_load_2d_at(dst + C::kTileB / 2, &a.tmap_b, bar, kb * C::kBK, a.N + n_blk * (BN / 2));
    }
  };
  // B is a weight, which no kernel of a step writes: its first stages are loaded while the
  // previous kernel still runs (kernel-level calls are launched after their predecessor's end).
  // Whole trajectories, without and with: tiny 666 / 651 us, DiT 5731 / 5685, SDXL 592 / 587, two
  // LLaDA blocks at 333 tokens 1090 / 1068 (one step each of U-ViT 1533 / 1526; level at 4096 rows).
  const int ahead = group < num_tiles ? min(kStages, a.num_k) : 0;
  if (warp == 0 && elect_one()) {
    int m_blk, n_blk;
    tile_coords(a, group, m_blk, n_blk);
    for (int kb = 0; kb < ahead; ++kb) load_b(n_blk, kb, kb);
  }
  __syncwarp();
  pdl_wait_and_trigger();  // the prologue above touched only shared memory, TMEM and B
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    const bool lead = elect_one();
    const uint32_t tiles0 = smem_u32(tiles), empty0 = smem_u32(empty);
    const uint32_t full0 = CG == 2 ? map_to_rank(smem_u32(full), 0) : smem_u32(full);  // the leader's barriers
    uint32_t st = 0, ph = 1;
    int it = 0;
    bool ok = true;
    for (int tile = group; tile < num_tiles && ok; tile += num_groups) {
      int m_blk, n_blk;
      tile_coords(a, tile, m_blk, n_blk);
      const int row_a = (CG * m_blk + static_cast<int>(rank)) * kBM;
      for (int kb = 0; kb < a.num_k; ++kb, ++it) {
        if (!mbar_wait_warp(empty0 + 8 * st, ph, abort_flag, a.status, 31)) {
          ok = false;
          break;
        }
        if (lead) {
          if (it >= ahead) load_b(n_blk, kb, st);
          const uint32_t bar = full0 + 8 * st, dst = tiles0 + st * kStageBytes;
          if constexpr (CG == 2)
            tma_load_2d_pair(dst, &a.tmap_a, bar, kb * C::kBK, row_a);
          else
            tma_load_2d_at(dst, &a.tmap_a, bar, kb * C::kBK, row_a);
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
        for (int i = tail; i < it; ++i) mbar_drain(&full[i % kStages], (i / kStages) & 1);
    } else if (lead) {
      // the releases committed to this CTA's barriers arrive before it ends
      for (int i = tail; i < it; ++i) mbar_drain(&empty[i % kStages], (i / kStages) & 1);
    }
  } else if (warp == 1) {
    if (rank == 0) {
      const bool lead = elect_one();
      constexpr uint32_t idesc = umma_idesc_f16(CG * kBM, BN);
      const uint32_t full0 = smem_u32(full), empty0 = smem_u32(empty);
      const uint64_t desc_a0 = smem_desc_sw128(smem_u32(tiles)), desc_b0 = smem_desc_sw128(smem_u32(tiles) + kTileA);
      uint64_t da = desc_a0, db = desc_b0;
      uint32_t st = 0, ph = 0;
      bool ok = true, ready = false;
      for (int tile = group, u = 0; tile < num_tiles && ok; tile += num_groups, ++u) {
        const int acc = u & 1;
        const uint32_t aph = (u >> 1) & 1;
        if (!mbar_wait_warp(smem_u32(&tempty[acc]), aph ^ 1u, abort_flag, a.status, 32)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * BN;
        uint32_t accumulate = 0;
        for (int kb = 0; kb < a.num_k; ++kb) {
          if (!ready && !mbar_wait_warp(full0 + 8 * st, ph, abort_flag, a.status, 33)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t bar = empty0 + 8 * st;
          if (lead) {
            umma_group<CG>(d_tmem, da, db, idesc, accumulate);
            umma_group<CG>(d_tmem, da + 2, db + 2, idesc, 1u);
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
            umma_group<CG>(d_tmem, ca + 4, cb + 4, idesc, 1u);
            umma_group<CG>(d_tmem, ca + 6, cb + 6, idesc, 1u);
            umma_commit_group<CG>(bar);
          }
        }
        if (!ok) break;
        if (lead) umma_commit_group<CG>(smem_u32(&tfull[acc]));
      }
      if (lead) umma_commit_group<CG>(smem_u32(drain));
    }
    // every MMA has finished, and the leader has committed for the last time, once `drain` completes
    if (lane == 0) mbar_drain(drain, 0);
  } else {
    float4* stg = reinterpret_cast<float4*>(tiles + kStages * kStageBytes + 512) + (warp - 2) * 256;
    const int q = warp & 3, part = (warp - 2) >> 2;
    constexpr int kSplit = ((BN / 32 + 1) / 2) * 32;
    const uint32_t tempty0 = CG == 2 ? map_to_rank(smem_u32(tempty), 0) : smem_u32(tempty);
    void* out = a.epi.out_slot ? *a.epi.out_slot : a.epi.out;
    float4 hv[8];  // first 32-column chunk of h (delta_staged)
    RopeTab rt;    // first chunk's tables (rope_staged)
    for (int tile = group, u = 0; tile < num_tiles; tile += num_groups, ++u) {
      int m_blk, n_blk;
      tile_coords(a, tile, m_blk, n_blk);
      const int acc = u & 1;
      const uint32_t aph = (u >> 1) & 1;
      const int row = (CG * m_blk + static_cast<int>(rank)) * kBM + q * 32 + lane;
      const uint32_t tbase = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + acc * BN;
      if (EP == kEpDelta) {
        prefetch_h_row(a.epi, row, a.M, a.N, n_blk * BN, part ? kSplit : 0, part ? BN : kSplit);
        load_h_chunk(a, row - lane, n_blk * BN + (part ? kSplit : 0), hv);
      }
      if (EP == kEpRope) rope_begin<BN>(a, row - lane, n_blk * BN, part, rt);
      if (!mbar_wait_warp(smem_u32(&tfull[acc]), aph, abort_flag, a.status, 34)) break;
      tc_fence_after();
      group_epilogue<BN, EP>(a, out, row, n_blk, TmemSrc{tbase, a.epi.alpha}, part, stg, hv, rt);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_leader<CG>(tempty0 + 8 * acc);
    }
  }

  tc_fence_before();
  __syncwarp();
  if constexpr (CG == 2)
    cluster_sync();  // nothing of either CTA refers to the other's memory any more
  else
    __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    if constexpr (CG == 2)
      tmem_dealloc_pair(tmem_base, C::kTmemCols);
    else
      tmem_dealloc(tmem_base, C::kTmemCols);
  }
}

template <int BN, int EP>
__global__ void __launch_bounds__(GroupCfg<1, BN>::kThreads, 1) gemm_one_kernel(const __grid_constant__ TcArgs a) {
  gemm_group_body<1, BN, EP>(a);
}
template <int BN, int EP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GroupCfg<2, BN>::kThreads, 1)
    gemm_pair_kernel(const __grid_constant__ TcArgs a) {
  gemm_group_body<2, BN, EP>(a);
}

template <int CG, int BN, int EP>
cudaError_t launch_group(const GemmPlan& p, const TcArgs& a, cudaStream_t s) {
  using C = GroupCfg<CG, BN>;
  void (*kernel)(const TcArgs);
  if constexpr (CG == 2)
    kernel = gemm_pair_kernel<BN, EP>;
  else
    kernel = gemm_one_kernel<BN, EP>;
  static bool attr_done[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr_done[dev]) {
    cudaError_t err = cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel),
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
    if (err != cudaSuccess) return err;
    attr_done[dev] = true;
  }
  return launch_k(kernel, dim3(p.grid), dim3(C::kThreads), C::kSmemBytes, s, a);
}

}  // namespace gk
}  // namespace sgd
