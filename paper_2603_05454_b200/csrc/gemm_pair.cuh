// bf16 GEMM on pairs of SMs (tcgen05.mma.cta_group::2), for passes of more than 128 activation rows.
//
//   acc[m, c] = sum_k A[m, k] * Wt[c, k]        operands and fused epilogues as k_gemm_stream (gemm_umma.cuh)
//
// With several row groups a layer GEMM is bound by the tensor pipe.  One SM working alone on a 128 x 256 tile takes in
// 48 KB per 64-element K atom; a cluster of two CTAs computing one 256 x BN tile takes in 32 KB per SM at BN = 256: each
// loads its own 128 activation rows and one half of the weight tile's BN rows (the MMA reads the other half from its peer)
// and keeps its own 128 accumulator rows in tensor memory.
//   * What bounds it otherwise is the producer and the issuer, one thread each: a turn of the stage ring (wait, arm, copies,
//     MMAs, commit) costs 300 ns whatever its size.  So a stage holds two K atoms and each operand of it is ONE copy (a 4-D
//     tensor map, see umma_map4), the MMAs of a stage share one commit, and whole warps run the loops with one elected
//     thread issuing (a lane branch around tcgen05.mma costs about 130 cycles per instruction, elect.sync 48 to 88).  With
//     one atom per stage and a copy per box the same kernel ran 4096 x 4096 outputs (K 4096) in 104 us, so 98, and
//     512 x 4096 in 25.3, so 17.8.
//   * Persistent: pair p takes every P-th tile (odd rounds in reverse order); the accumulators are double-buffered (2 x BN of 512 columns), so the
//     epilogue of a tile overlaps the next tile's MMAs.
//   * A last row group of at most 128 rows runs on 128-row MMAs (see pair_half_last).
//   * BN is a run-time multiple of 32 (64 for the rotary epilogue), the one with the least time by a model of a pair's
//     intake over all rounds (see pair_shape); whole tiles are dealt, so the last round may still leave pairs idle.
//   * The weight tile's two halves come from the two tensors / row ranges whose columns a fused epilogue pairs (gate and
//     up, rotate-half partners), so CTA 0 always loads the first and CTA 1 the second of the pair.
//   * Eight epilogue warps: two per quarter of the accumulator rows, each taking half of the 16-column chunks.  The
//     residual epilogue fetches its rows of x while it waits for the accumulators.
// Measured (B200, back to back, weights from a ring larger than L2; one SM per tile before -> now, us):
//   rows    12288 x 4096   4096 x 4096   2 x 12288 x 4096 SwiGLU   4096 x 12288
//    512      58 -> 42      31 -> 17            111 -> 76          56 -> 45
//   1000     104 -> 74      41 -> 28            153 -> 139          86 -> 75
//   4096     313 -> 271     129 -> 99            559 -> 512         311 -> 297
//   8240     646 -> 551     260 -> 202           1205 -> 1050        657 -> 596
// Warp roles (320 threads): warp 0 = TMA producer, warp 1 = TMEM allocator and, in the pair's first CTA, MMA issuer,
// warps 2..9 = epilogue.  Every wait is bounded; on expiry the kernel records (code, site) in the status word, drains and
// returns.
#pragma once
#include <algorithm>

#include "gemm_stream.cuh"

namespace lsp {

constexpr int PR_THREADS = 320;
constexpr int PR_MAX_STAGES = 8;
constexpr int PR_ROWS = 256;               // activation rows per tile

struct PairArgs {
  int M;            // activation rows
  int n_pairs;      // dual: pair indices; plain: output columns
  int n_tiles;      // column tiles
  int row_groups;   // groups of 256 activation rows
  int band;         // row groups per band: tiles are ordered band by band, within a band column tile by column tile
  int kc;           // chunks of 128 K elements (two atoms; the last one may be half empty: zero-filled)
  int ks;           // K slices of a tile (plain epilogues, one tile per cluster): pair s of the cluster takes the s-th share of
                    // the chunks, and the partial tiles are summed through distributed shared memory
  int bn;           // tile width
  int chains;       // head with one tile per pair: accumulators that take K in turn (see umma_head_shape), else 1
  int half_last;    // the last row group has at most 128 rows and runs with 128-row MMAs (64 rows per CTA)
  int unit;         // rotary epilogue: 0 where a half tile is made of whole head halves; else 32, and tiles 2 g and 2 g + 1 are the first and
                    // the second 32 frequencies of bn / 64 heads: one copy brings such rows of several heads, where a tile of
                    // consecutive pairs would take one per 32 rows and K atom (six a stage at 192 columns: 12288 x 4096 with 512 rows
                    // took 57 us where the same tiles of a plain epilogue take 42; LLaDA-shaped passes of 187 / 512 rows 4.87 ->
                    // 4.80, 7.93 -> 7.77 ms)
  int stages;
  unsigned* status;
};

// One box of a 4-D map (umma_map4) into this CTA's shared memory; the bytes are counted on the barrier `bar` (a
// shared::cluster address: the barrier of the pair's first CTA).
__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap* map, int r0, int blk, int a0, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(map), "r"(0), "r"(r0), "r"(blk), "r"(a0), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tc_mma_f16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrives at the barrier at this offset in both CTAs of the pair (mask: their cluster ranks) once the issued MMAs have completed
__device__ __forceinline__ void tc_commit_pair(uint32_t bar, uint16_t mask) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"(mask)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

template <typename Epi>
__global__ void __launch_bounds__(PR_THREADS, 1)
k_gemm_pair(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b0,
            const __grid_constant__ CUtensorMap map_b1, const __grid_constant__ CUtensorMap map_ah,
            const __grid_constant__ CUtensorMap map_h0, const __grid_constant__ CUtensorMap map_h1, PairArgs args, Epi epi) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int A_ATOM = UM_BM * 128;                     // this CTA's 128 activation rows of one K atom
  constexpr uint32_t TMEM_COLS = 512;
  constexpr bool kRope = std::is_same<Epi, EpiQKVRope<bf16>>::value;
  if (!kRope) pdl_release();
  const int BN = args.bn, HALF = BN / 2;
  const int B_ATOM = HALF * 128;
  const int STAGE_BYTES = 2 * (A_ATOM + B_ATOM);          // two K atoms
  const int S = args.stages;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)S * STAGE_BYTES);
  // bars[0..S) full (used in the first CTA), [S..2S) empty, [2S..2S+2) accumulators full, [2S+2..2S+4) accumulators empty
  // (used in the first CTA)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 4);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar_base = smem_u32(bars);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (S + s); };
  auto accf_bar = [&](int b) { return bar_base + 8u * (2 * S + b); };
  auto acce_bar = [&](int b) { return bar_base + 8u * (2 * S + 2 + b); };

  const int crank = (int)cluster_ctarank(), rank = crank & 1;           // rank within the pair
  const unsigned lead = (unsigned)(crank & ~1);                           // the pair's first CTA
  const int ks = args.ks, slice = crank >> 1;
  const uint16_t pair_mask = (uint16_t)(3u << lead);
  const int P = gridDim.x / (unsigned)(2 * ks), pair = blockIdx.x / (unsigned)(2 * ks);
  const int T = args.n_tiles * args.row_groups;
  // tiles are dealt in rounds, odd rounds in reverse, so that with an even number of row groups a pair gets some of each
  const int rest = T % P;
  const int my_tiles = T / P + ((((T / P) & 1) ? P - 1 - pair : pair) < rest ? 1 : 0);      // the host launches at most T pairs
  const int kc0 = args.kc * slice / ks, kc = args.kc * (slice + 1) / ks - kc0;      // this pair's chunks
  const int n_units = my_tiles * kc;
  // i-th tile of this pair -> column tile and row group
  auto tile_of = [&](int i, int& tile, int& rg) {
    const int t = i * P + ((i & 1) ? P - 1 - pair : pair);
    const int per_band = args.band * args.n_tiles;
    const int b = t / per_band, r = t - b * per_band;
    const int rows = min(args.band, args.row_groups - b * args.band);
    tile = r / rows;
    rg = b * args.band + r % rows;
  };
  const uint32_t full0 = cluster_map(bar_base, lead);     // the first CTA's full barriers, in the cluster's window
  constexpr bool kHalf = !kRope && !Epi::kReduce;
  auto half_rows = [&](int rg) { return kHalf && args.half_last && rg == args.row_groups - 1; };
  const CUtensorMap* map_b = rank ? &map_b1 : &map_b0;    // this CTA's half of the weight tile
  auto load_weights = [&](int tile, int rg, int c, int s) {
    const uint32_t sb = smem_u32(smem + (size_t)s * STAGE_BYTES) + 2 * A_ATOM;
    if constexpr (kRope) {
      // blocks of the map are head halves
      if (args.unit == 0) tma_load_4d_pair(sb, map_b, 0, tile * HALF / epi.half, 2 * c, full0 + 8u * s);
      else tma_load_4d_pair(sb, map_b, (tile & 1) * 32, (tile >> 1) * (HALF / 32), 2 * c, full0 + 8u * s);
    } else if (Epi::kDual && half_rows(rg)) {
      // the MMA leaves columns [0, HALF) in lanes 0 .. 63 and [HALF, BN) in lanes 64 .. 127: this CTA's half of the weight tile
      // is then the rank-th half of the tile's gate rows and the same of its up rows, so that a pair stays in one lane
      const int j = tile * HALF + rank * (HALF / 2);
      for (int a = 0; a < 2; ++a) {
        tma_load_4d_pair(sb + a * B_ATOM, &map_h0, j, 0, 2 * c + a, full0 + 8u * s);
        tma_load_4d_pair(sb + a * B_ATOM + B_ATOM / 2, &map_h1, j, 0, 2 * c + a, full0 + 8u * s);
      }
    } else {
      tma_load_4d_pair(sb, map_b, Epi::kDual ? tile * HALF : tile * BN + rank * HALF, 0, 2 * (kc0 + c), full0 + 8u * s);
    }
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf_bar(b), 1);
      mbar_init(acce_bar(b), 16);           // eight epilogue warps of each CTA
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();                            // both CTAs' barriers and tensor memory are set up
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const int n_pre = n_units < S ? n_units : S;
    int tile = 0, rg = 0, c = 0, i = 0;
    tile_of(0, tile, rg);
    // weights are never written by any kernel: the first stages' are requested while the preceding kernel still runs
    {
      int t2 = tile, rg2 = rg, c2 = 0, i2 = 0;
      for (int it = 0; it < n_pre; ++it) {
        if (elect_one()) {
          if (rank == 0) mbar_expect_tx(full_bar(it), half_rows(rg2) ? 2 * STAGE_BYTES - 2 * A_ATOM : 2 * STAGE_BYTES);
          load_weights(t2, rg2, c2, it);
        }
        __syncwarp();
        if (++c2 == kc) { c2 = 0; if (++i2 < my_tiles) tile_of(i2, t2, rg2); }
      }
    }
    pdl_wait();
    if (kRope) pdl_release();        // the attention that follows reads older keys and values ahead of its own wait
    int s = 0, issued = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int it = 0; it < n_units; ++it) {
      if (it >= n_pre) {
        ok = __all_sync(0xffffffffu, mbar_wait(empty_bar(s), ph ^ 1u, abort_flag));
        if (!ok) {
          if (lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(args.status, 1u); args.status[1] = 41u; }
          break;
        }
      }
      if (elect_one()) {
        if (it >= n_pre) {
          if (rank == 0) mbar_expect_tx(full_bar(s), half_rows(rg) ? 2 * STAGE_BYTES - 2 * A_ATOM : 2 * STAGE_BYTES);
          load_weights(tile, rg, c, s);
        }
        if (half_rows(rg))
          tma_load_4d_pair(smem_u32(smem + (size_t)s * STAGE_BYTES), &map_ah, rg * PR_ROWS + rank * 64, 0, 2 * (kc0 + c), full0 + 8u * s);
        else
          tma_load_4d_pair(smem_u32(smem + (size_t)s * STAGE_BYTES), &map_a, rg * PR_ROWS + rank * UM_BM, 0, 2 * (kc0 + c), full0 + 8u * s);
      }
      __syncwarp();
      ++issued;
      if (++s == S) { s = 0; ph ^= 1u; }
      if (++c == kc) { c = 0; if (++i < my_tiles) tile_of(i, tile, rg); }
    }
    // do not leave while copies may still be landing: the first CTA's barriers count both CTAs' copies, and the cluster
    // barrier at the end holds the second CTA until the first has seen them
    volatile uint32_t no_abort = 0;
    if (rank == 0) {
      for (int it = issued > S ? issued - S : 0; it < issued; ++it) mbar_wait(full_bar(it % S), (uint32_t)(it / S) & 1u, &no_abort);
    }
    if (!ok) um_let_land();                // (the peer may not have counted these copies)
  } else if (warp == 1) {
    // ---------------- MMA issuer (first CTA; the whole warp waits, one elected thread issues) ----------------
    pdl_wait();            // (its bounded waits must not count the preceding kernel's time)
    if (rank == 0) {
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int i = 0; i < my_tiles && ok; ++i) {
        const int buf = i & 1, use = i >> 1;
        int tile, rg;
        tile_of(i, tile, rg);
        const bool half = half_rows(rg);
        const uint32_t idesc = (make_idesc(BN) & ~(31u << 24)) | ((uint32_t)((half ? PR_ROWS / 2 : PR_ROWS) >> 4) << 24);
        const uint32_t a_atom = half ? A_ATOM / 2 : A_ATOM;
        if (use >= 1) ok = mbar_wait(acce_bar(buf), (uint32_t)(use - 1) & 1u, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
          if (lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(args.status, 1u); args.status[1] = 42u; }
          break;
        }
        tc_fence_after();
        uint32_t d = tmem_base + (uint32_t)(buf * 256), acc = 0;              // acc 0: the next MMA overwrites the accumulator
        int chain = 0, chain_end = 2 * kc / args.chains;                      // (in K atoms)
        for (int c = 0; c < kc; ++c) {
          ok = mbar_wait(full_bar(s), ph, abort_flag);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) {
            if (lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(args.status, 1u); args.status[1] = 43u; }
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + (size_t)s * STAGE_BYTES);
          if (elect_one()) {
#pragma unroll
            for (int a = 0; a < 2; ++a) {
              if (Epi::kReduce && 2 * c + a == chain_end) {
                chain_end = 2 * kc * (++chain + 1) / args.chains;
                d += (uint32_t)BN;
                acc = 0;
              }
              const uint64_t da = make_smem_desc(sa + a * a_atom), db = make_smem_desc(sa + 2 * A_ATOM + a * B_ATOM);
#pragma unroll
              for (int k = 0; k < 4; ++k)
                tc_mma_f16_pair(d, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc, acc | (uint32_t)k ? 1u : 0u);
              acc = 1;
            }
            tc_commit_pair(empty_bar(s), pair_mask);
            if (c == kc - 1) tc_commit_pair(accf_bar(buf), pair_mask);
          }
          __syncwarp();
          if (++s == S) { s = 0; ph ^= 1u; }
        }
      }
    }
  } else {
    // ---------------- epilogue ----------------
    pdl_wait();
    const int q = warp & 3;                                       // the quarter of tensor-memory lanes this warp may read
    const int h = (warp - 2) >> 2;                                // column half
    const int r_in = q * 32 + lane;
    const int CH = Epi::kDual ? HALF : BN;                        // pair indices (dual) or columns (plain) per tile
    const uint32_t acce0 = cluster_map(acce_bar(0), lead);
    for (int i = 0; i < my_tiles && ks == 1; ++i) {
      const int buf = i & 1, use = i >> 1;
      int tile, rg;
      tile_of(i, tile, rg);
      const bool half = half_rows(rg);                            // 64 rows per CTA, lanes 64 .. 127: the second half of the columns
      const int m = half ? rg * PR_ROWS + rank * 64 + (r_in & 63) : rg * PR_ROWS + rank * UM_BM + r_in;
      const int j0 = tile * CH + (half && q >= 2 ? CH / 2 : 0);
      const int nch = half ? CH >> 5 : CH >> 4, mid = (nch + 1) >> 1;
      const int ch_lo = h ? mid : 0, ch_hi = h ? nch : mid;
      const uint32_t up = (uint32_t)(half ? HALF / 2 : HALF);     // dual: the second accumulator's first column
      const bool live = m < args.M;
      uint4 xr[16];
      if constexpr (std::is_same<Epi, EpiResidual<bf16>>::value) {
        // this thread's part of the residual rows, fetched while the MMAs run
        const uint4* xp = reinterpret_cast<const uint4*>(epi.x + (size_t)m * epi.ld + j0 + ch_lo * 16);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (live && ch_lo + k < ch_hi && j0 + (ch_lo + k) * 16 < args.n_pairs) {
            xr[2 * k] = xp[2 * k];
            xr[2 * k + 1] = xp[2 * k + 1];
          }
        }
      }
      // rotary table entries of the first two chunks, fetched while the MMAs run, then two chunks ahead (fetched behind the last MMA,
      // one ahead: LLaDA-shaped passes of 187 / 512 rows 5.14 -> 5.04, 8.12 -> 8.04 ms)
      EpiPre<Epi> pre, next;
      auto pair_at = [&](int ch) {                                // pair index of a chunk
        if (kRope && args.unit) return ((tile >> 1) * (HALF / 32) + (ch >> 1)) * 64 + (tile & 1) * 32 + (ch & 1) * 16;
        return j0 + ch * 16;
      };
      auto fetch = [&](int ch, EpiPre<Epi>& p) {
        if (live && ch < ch_hi && pair_at(ch) < args.n_pairs) p.load(epi, m, pair_at(ch));
      };
      if constexpr (kRope) {
        fetch(ch_lo, pre);
        fetch(ch_lo + 1, next);
      }
      if (!__all_sync(0xffffffffu, mbar_wait(accf_bar(buf), (uint32_t)use & 1u, abort_flag))) {
        if (lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(args.status, 1u); args.status[1] = 44u; }
        break;
      }
      tc_fence_after();
      const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 256);
      if constexpr (std::is_same<Epi, EpiResidual<bf16>>::value) {
        uint4* xp = reinterpret_cast<uint4*>(epi.x + (size_t)m * epi.ld + j0 + ch_lo * 16);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (ch_lo + k < ch_hi) {                                // uniform per warp
            float a[16];
            __syncwarp();                                         // (rows past the last one part ways above; the load is collective)
            tc_ld16(t_row + (uint32_t)((ch_lo + k) * 16), a);
            if (live && j0 + (ch_lo + k) * 16 < args.n_pairs) {
#pragma unroll
              for (int hh = 0; hh < 2; ++hh) {
                float x[8];
                unpack8(xr[2 * k + hh], x);
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] += a[8 * hh + e];
                xp[2 * k + hh] = pack8(x);
              }
            }
          }
        }
      } else {
        Top2 red = top2_empty();
        auto consume = [&](int ch, float (&a0)[16], float (&a1)[16]) {
          const int j = j0 + ch * 16;
          if constexpr (Epi::kReduce) top2_push16(red, a0, j, epi);
          else if (live && j < args.n_pairs) epi16(epi, m, j, a0, a1);
          __syncwarp();                                           // (rows past the last one part ways above; the next load is collective)
        };
        auto request = [&](int ch, float (&a0)[16], float (&a1)[16]) {
          tc_ld16_nowait(t_row + (uint32_t)(ch * 16), a0);
          if (Epi::kDual) tc_ld16_nowait(t_row + up + (uint32_t)(ch * 16), a1);
        };
        if constexpr (kRope) {
          // (the rotary table's entries ahead take the registers a second set of accumulator values would)
          float p0[16], p1[16];
#pragma unroll 1
          for (int ch = ch_lo; ch < ch_hi; ++ch) {
            __syncwarp();
            request(ch, p0, p1);
            tc_wait_ld();
            tc_pin16(p0);
            tc_pin16(p1);
            if (live && pair_at(ch) < args.n_pairs) epi16(epi, m, pair_at(ch), p0, p1, pre);
            pre = next;
            fetch(ch + 2, next);
          }
        } else if (Epi::kReduce && args.chains > 1) {
#pragma unroll 1
          for (int ch = ch_lo; ch < ch_hi; ++ch) {
            float sum[16], part[16];
            tc_ld16(t_row + (uint32_t)(ch * 16), sum);
#pragma unroll 1
            for (int x = 1; x < args.chains; ++x) {
              tc_ld16(t_row + (uint32_t)(x * BN + ch * 16), part);
#pragma unroll
              for (int e = 0; e < 16; ++e) sum[e] += part[e];
            }
            consume(ch, sum, part);
          }
        } else {
        // the next chunk's tensor-memory loads are in flight while this one is converted and stored
        float p0[16], p1[16], q0[16], q1[16];
        if (ch_lo < ch_hi) request(ch_lo, p0, p1);
#pragma unroll 1
        for (int ch = ch_lo; ch < ch_hi; ch += 2) {
          tc_wait_ld();
          tc_pin16(p0);
          if (Epi::kDual) tc_pin16(p1);
          if (ch + 1 < ch_hi) request(ch + 1, q0, q1);
          consume(ch, p0, p1);
          if (ch + 1 < ch_hi) {
            tc_wait_ld();
            tc_pin16(q0);
            if (Epi::kDual) tc_pin16(q1);
            if (ch + 2 < ch_hi) request(ch + 2, p0, p1);
            consume(ch + 1, q0, q1);
          }
        }
        }
        if constexpr (Epi::kReduce) {
          if (live) epi.part[(size_t)m * epi.n_tiles + 2 * tile + h] = red;      // one partial per column half
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acce0 + 8u * buf);
    }
  }
  if constexpr (!Epi::kDual && !Epi::kReduce) {
    if (ks > 1) {
      // K slices: the pair of slice s finishes the s-th share of the tile's 16-column chunks.  Every CTA publishes the other
      // shares of its 128 rows in its own shared memory (the pipeline stages are idle once the accumulator is complete), and
      // after a cluster barrier adds, for its own share, the pieces of the other slices' CTAs with the same rows to its own,
      // in slice (= K) order.  All threads of all CTAs reach both barriers.
      const int q = warp & 3, h = (warp - 2) >> 2, r_in = q * 32 + lane, nch = BN >> 4;
      const int lo = nch * slice / ks, hi = nch * (slice + 1) / ks;                 // this slice's chunks
      int tile, rg;
      tile_of(0, tile, rg);
      const int m = rg * PR_ROWS + rank * UM_BM + r_in, j0 = tile * BN;
      const bool live = m < args.M;
      const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16);
      float4* pub = reinterpret_cast<float4*>(smem);                               // [chunk][quarter][row]
      bool ok = true;
      if (warp >= 2) {
        ok = __all_sync(0xffffffffu, mbar_wait(accf_bar(0), 0u, abort_flag));
        if (!ok && lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(args.status, 1u); args.status[1] = 45u; }
        tc_fence_after();
        if (ok) {
          for (int ch = h; ch < nch; ch += 2) {                                     // the two warps of a quarter alternate
            if (ch >= lo && ch < hi) continue;
            float v[16];
            __syncwarp();
            tc_ld16(t_row + (uint32_t)(ch * 16), v);
            if (live) {
#pragma unroll
              for (int g = 0; g < 4; ++g) pub[(ch * 4 + g) * UM_BM + r_in] = make_float4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
            }
          }
        }
      }
      EpiPre<Epi> pre;
      if (warp >= 2 && live && lo + h < hi && j0 + (lo + h) * 16 < args.n_pairs) pre.load(epi, m, j0 + (lo + h) * 16);
      cluster_sync();
      if (warp >= 2 && ok) {
        for (int ch = lo + h; ch < hi; ch += 2) {
          float own[16], a[16];
          __syncwarp();
          tc_ld16(t_row + (uint32_t)(ch * 16), own);
          if (live && j0 + ch * 16 < args.n_pairs) {
            float4 t[2][4];                                                        // (at most three slices)
#pragma unroll
            for (int x = 0; x < 2; ++x) {
              const int p = x < slice ? x : x + 1;
              if (p < ks) {
                const uint32_t peer = cluster_map(smem_u32(smem), (unsigned)(2 * p + rank)) + (uint32_t)((ch * 4 * UM_BM + r_in) * 16);
#pragma unroll
                for (int g = 0; g < 4; ++g) t[x][g] = ld_cluster_f4(peer + (uint32_t)(g * UM_BM * 16));
              }
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) a[i] = 0.f;
#pragma unroll
            for (int p = 0; p < 3; ++p) {
              if (p >= ks) break;
              if (p == slice) {
#pragma unroll
                for (int i = 0; i < 16; ++i) a[i] += own[i];
              } else {
                const int x = p < slice ? p : p - 1;
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                  const float4 u = x == 0 ? t[0][g] : t[1][g];
                  a[4 * g] += u.x; a[4 * g + 1] += u.y; a[4 * g + 2] += u.z; a[4 * g + 3] += u.w;
                }
              }
            }
            epi16(epi, m, j0 + ch * 16, a, a, pre);
            if (ch + 2 < hi && j0 + (ch + 2) * 16 < args.n_pairs) pre.load(epi, m, j0 + (ch + 2) * 16);
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();          // nobody leaves while its peer may still read its shared memory or signal its barriers
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// ---- host side ------------------------------------------------------------------------------------------------
// Tile width and K slices.  What a chunk of 128 K elements costs a pair is its intake: 32 KB of activations and bn / 8 KB of
// weights per SM at about 118 GB/s from L2, i.e. 1.06 ns x (bn + 256), which the MMAs of the widest tile just fill.  (Under the
// power cap, with many rounds, bn + 44 fits better: per 4096 K elements 11.4 / 13.5 / 16.1 / 18.9 / 21.8 / 24.6 us at 96 / 128 /
// 160 / 192 / 224 / 256 columns.)  A launch takes as many rounds as its fullest pair.  A plain projection whose tiles fit
// once with two or three K slices each may split: wider tiles re-read the activations less, at 10 to 14 us for the exchange
// (187 rows, 4096 x 12288: 34.6 us whole, 28.5 in three slices; 3584 x 18944: 48.2, 35.5; but 512 rows, 4096 x 12288: 45.0 whole,
// 47.9 in two).
// step: widths are multiples of 32, or 64 for the rotary epilogue (a half tile is then made of whole 32-row boxes inside one
// head half).
struct PairShape { int bn, ks; };
// A last row group of at most 128 rows runs with 128-row MMAs (64 rows per CTA, which leave the tile's column halves in the two
// halves of the lanes): 24 KB instead of 32 per SM and K atom at 256 columns and half the tensor work, about 0.75 of a tile's
// time.
// 1032 rows, 2 x 18944 x 3584: 222.5 -> 209.4 us; 3584 x 18944: 116.5 -> 114.5; 300 rows, 4096 x 12288: 43.4 -> 41.5, 4096 x 4096: 17.3
// -> 16.5, 2 x 12288 x 4096 (now 256 columns wide): 74.8 -> 68.6.  The epilogues whose columns cannot be halved that way (rotary
// pairs inside a head, the head's partials per tile half) and widths that are no multiple of 64 keep 256-row MMAs.
inline bool pair_half_last(int M, int bn) {
  const int last = M % PR_ROWS;
  return M > PR_ROWS && last >= 1 && last <= PR_ROWS / 2 && bn % 64 == 0;
}
// Column tiles of width bn.  rot_half: pair indices per head of a rotary epilogue (else 0); where a half tile is no whole head halves, two
// tiles are the halves of bn / 64 heads (see PairArgs::unit), and the last two may stand for fewer.
inline int pair_tiles(int cols, int bn, int rot_half) {
  if (rot_half == 0 || bn / 2 % rot_half == 0) return (cols + bn - 1) / bn;
  const int heads = cols / (2 * rot_half), nb = bn / 64;
  return (heads + nb - 1) / nb * 2;
}
inline PairShape pair_shape(const UmmaState& st, int M, int cols, int K, int step, bool may_split, bool may_halve, int rot_half) {
  const int pairs = st.max_clusters[2];
  const long rg = (M + PR_ROWS - 1) / PR_ROWS;
  const double chunks = (K + 127) / 128;
  PairShape best{256, 1};
  double best_cost = 1e30;
  for (int bn = 256; bn >= 96; bn -= step) {
    const long t = (long)pair_tiles(cols, bn, rot_half) * rg;
    const long rounds = (t + pairs - 1) / pairs;
    const double share = (may_halve && pair_half_last(M, bn)) ? (rg - 0.25) / rg : 1.0;     // of a full tile's time
    const double cost = share * chunks * (rounds > 2 ? rounds * (bn + 44) * 1.8 : rounds * (bn + 256)) * 1.06e-3;
    if (cost < best_cost - 1e-9) { best_cost = cost; best = {bn, 1}; }
    for (int ks = 2; ks <= 3 && may_split; ++ks) {
      if (t * ks > pairs || t > st.max_clusters[2 * ks] || chunks < 8 * ks) continue;
      const double c2 = chunks / ks * (bn + 256) * 1.06e-3 + 14.0;
      if (c2 < best_cost - 1e-9) { best_cost = c2; best = {bn, ks}; }
    }
  }
  return best;
}

template <typename Epi>
int pair_launch(UmmaState& st, cudaStream_t stream, const bf16* A, const bf16* W0, const bf16* W1, int M, int NP, int K,
                int n_rows_w, const Epi& epi, unsigned* status) {
  constexpr bool kRope = std::is_same<Epi, EpiQKVRope<bf16>>::value;
  const int cols = Epi::kDual ? 2 * NP : NP;
  const int pairs = st.max_clusters[2];
  constexpr bool kPlain = !Epi::kDual && !Epi::kReduce;
  PairShape shape{UM_HEAD_BN, 1};
  int chains = 1, rot_half = 0;
  if constexpr (kRope) rot_half = epi.half;
  if constexpr (Epi::kReduce) {
    const HeadShape h = umma_head_shape(st, M, NP, K);
    shape.bn = h.bn;
    chains = std::min(h.chains, K / UM_BK);
  } else {
    shape = pair_shape(st, M, cols, K, kRope ? 64 : 32, kPlain && st.pair_split != 1, !kRope, rot_half);
    if (st.pair_bn > 0 && (!kRope || st.pair_bn % 64 == 0)) shape = {st.pair_bn, 1};      // (a width that the epilogue can take)
  }
  const int bn = shape.bn;
  int unit = 0;
  if constexpr (kRope) {
    if ((bn / 2) % epi.half) unit = 32;
    // a half tile is whole boxes, each inside one head half: a box too many would land behind its stage
    if (epi.half % 32 || bn % 64) { st.err = "unsupported head_dim or tile width for the paired GEMM's rotary epilogue"; return -6; }
  }
  const int stage = 2 * (UM_BM * 128 + bn / 2 * 128);
  const int aux = 1024 + 8 * (2 * PR_MAX_STAGES + 4) + 16;
  int stages = (st.max_smem - aux) / stage;
  if (stages > PR_MAX_STAGES) stages = PR_MAX_STAGES;
  if (stages < 2) { st.err = "not enough shared memory for the paired GEMM"; return -2; }
  const size_t smem = (size_t)stages * stage + aux;
  const cudaError_t smem_rc = umma_raise_smem(st, k_gemm_pair<Epi>);
  if (smem_rc != cudaSuccess) { st.err = cudaGetErrorString(smem_rc); return -3; }
  CUtensorMap ma, mb0, mb1, mah, mh0, mh1;               // ..h: operands of a half row group
  const int half_last = (!kRope && !Epi::kReduce && shape.ks == 1 && st.pair_split <= 1 && pair_half_last(M, bn)) ? 1 : 0;
  {
    const CUtensorMap* p = umma_map4(st, A, M, M, 1, K, UM_BM, 1, 2);
    if (!p) return -4;
    ma = *p;
    if constexpr (kRope) {
      const int blocks = n_rows_w / (2 * epi.half), br = unit ? unit : epi.half, bb = bn / 2 / br;
      p = umma_map4(st, W0, epi.half, 2 * epi.half, blocks, K, br, bb, 2);
      if (!p) return -4;
      mb0 = *p;
      p = umma_map4(st, W1 + (size_t)epi.half * K, epi.half, 2 * epi.half, blocks, K, br, bb, 2);
    } else {
      p = umma_map4(st, W0, n_rows_w, n_rows_w, 1, K, bn / 2, 1, 2);
      if (!p) return -4;
      mb0 = *p;
      p = umma_map4(st, W1, n_rows_w, n_rows_w, 1, K, bn / 2, 1, 2);
    }
    if (!p) return -4;
    mb1 = *p;
    mah = ma;
    mh0 = mb0;
    mh1 = mb1;
    if (half_last) {
      p = umma_map4(st, A, M, M, 1, K, UM_BM / 2, 1, 2);
      if (!p) return -4;
      mah = *p;
      if (Epi::kDual) {
        p = umma_map4(st, W0, n_rows_w, n_rows_w, 1, K, bn / 4, 1, 1);
        if (!p) return -4;
        mh0 = *p;
        p = umma_map4(st, W1, n_rows_w, n_rows_w, 1, K, bn / 4, 1, 1);
        if (!p) return -4;
        mh1 = *p;
      }
    }
  }
  const int n_tiles = pair_tiles(cols, bn, rot_half);
  const int rg = (M + PR_ROWS - 1) / PR_ROWS;
  const long T = (long)n_tiles * rg;
  if (T > (1l << 24)) { st.err = "too many tiles for the paired GEMM"; return -9; }
  // Bands of row groups whose activation rows (at most about 40 MB) stay in L2 while the weights stream past them once per
  // band: 8240 x 12288 x 2 (K 4096) 1146 us in one band, 1067 in bands of 16; 8240 x 4096 (K 12288) 648 in one, 589 in bands
  // of 4, 751 in bands of 2 (then the weights, streamed too often, are the larger part).
  int band_max = (int)(40e6 / ((double)PR_ROWS * K * 2));
  if (band_max < 4) band_max = 4;
  if (st.pair_band > 0) band_max = st.pair_band;
  const int n_bands = (rg + band_max - 1) / band_max, band = (rg + n_bands - 1) / n_bands;
  int ks = shape.ks;
  if (kPlain && st.pair_split > 1 && T * st.pair_split <= pairs && T <= st.max_clusters[2 * st.pair_split] && (K + 127) / 128 >= st.pair_split)
    ks = st.pair_split;
  const int grid = 2 * ks * (int)(T < pairs ? T : pairs);
  PairArgs args{M, NP, n_tiles, rg, band, (K + 2 * UM_BK - 1) / (2 * UM_BK), ks, bn, chains, half_last, unit, stages, status};
  cudaError_t e = launch_k(st.pdl, k_gemm_pair<Epi>, dim3(grid), dim3(PR_THREADS), smem, stream, 2 * ks, ma, mb0, mb1, mah, mh0, mh1, args, epi);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) { st.err = cudaGetErrorString(e); return -5; }
  return 0;
}

}  // namespace lsp
