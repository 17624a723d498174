// Persistent bf16 GEMM on tcgen05 for the weight-streaming regime: at most 128 activation rows (the shrinking suffix of late
// decode steps; more rows go to the pairs of SMs, gemm_pair.cuh).
//
//   acc[m, c] = sum_k A[m, k] * Wt[c, k]        operands, descriptors and fused epilogues: gemm_umma.cuh
//
// Such a GEMM is bound by reading its weights from HBM once, so the kernel is built around one uninterrupted stream of weight
// tiles per SM:
//   * persistent CTAs, at most one per SM; the (column tile, K chunk) units of the whole problem are dealt out in
//     equal contiguous shares (a share may start and end in the middle of a tile), in a single wave;
//   * a pipeline stage holds 128 elements of K (two 128-byte swizzle atoms per operand) when at least three such
//     stages fit, else 64: 256 contiguous bytes per weight row and stage stream at 5.3 TB/s on B200 where 128 bytes
//     per row and stage reach only 3.7 TB/s;
//   * only the activation rows that exist are loaded (a box of M rounded up to 8 rows); the MMAs still span 128
//     accumulator rows, and the rows past the box, computed from whatever the stage holds, are never stored;
//   * accumulators are double-buffered in tensor memory, so the epilogue of one tile overlaps the loads and MMAs of the next;
//     only the first fill and the last epilogue of a CTA are exposed;
//   * the K slices of a split tile form a cluster and are reduced through distributed shared memory; without clusters (the
//     head, whose tiles outnumber the SMs) a tile that spans several CTAs is finished by the one that arrives last at the
//     tile's counter: every contributor writes its fp32 partial tile to scratch, and the finisher sums all of them in CTA order
//     (the same order whoever finishes, so results are deterministic) before running the fused epilogue.
// Tile width: measured per shape and row count (see umma_gemm): 128 columns for plain epilogues (no K split needed with 96
// tiles), 256 or 192 for dual ones.
// Producer and issuers are whole warps with one elected thread issuing, and each operand of a stage is one copy (4-D and 5-D
// tensor maps, gemm_umma.cuh): against a lane branch and a copy per half tile and K atom 2 x 12288 x 4096 SwiGLU at 101 rows
// 38.7 -> 35.5 us, 12288 x 4096 25.7 -> 24.7, 3584 x 18944 at 9 rows 28.8 -> 26.4; a LLaDA-shaped pass of 9 rows
// 4.20 -> 3.95 ms, of 101 rows 4.82 -> 4.51.
// The activations have a producer of their own: where the preceding kernel has just ended (the O and down projections start when
// its CTAs leave the SMs) their first request would queue behind the 200 KB of weights that fill the ring, and the first MMA came 5 us
// after the launch's start instead of 3 (a LLaDA-shaped pass of 9 rows 3.74 -> 3.63 ms, of 101 rows 4.28 -> 4.19).  And the issuer looks at
// the next stage between this one's MMAs: waiting for it behind the commit leaves the tensor pipe empty meanwhile (8 MMAs of 128 columns
// 749 -> 659 cycles a stage; the passes another 2 to 4 %).
// Warp roles (224 threads): warp 0 = TMA producer of the weights, warp 6 = of the activations, warp 1 = TMEM allocator + MMA issuer,
// warps 2..5 = epilogue.
// Every wait is bounded; on expiry the kernel records (code, site) in the status word, drains and returns.
#pragma once
#include <algorithm>

#include "cluster.cuh"
#include "gemm_umma.cuh"

namespace lsp {

constexpr int ST_MAX_STAGES = 8;

struct StreamArgs {
  int M;            // activation rows (<= 128)
  int n_pairs;      // dual: pair indices; plain: output columns
  int n_tiles;      // column tiles
  int cluster;      // > 1: the launch uses thread block clusters of this size, one cluster per tile, CTA rank r owning the
                    // r-th K slice; the partial tiles are then reduced through distributed shared memory (see the kernel)
  int exchange;     // clusters of 2: each CTA publishes only the half its peer finishes and keeps its own half in tensor memory
  int kc;           // K chunks (one per stage) per tile
  int chains;       // rotary epilogue, one whole tile per CTA: accumulators that take K in turn, added in K order (else 1)
  int a_rows;       // activation box rows (M rounded up to a multiple of 8)
  int atoms;        // 64-element K atoms per stage (1 or 2)
  int one_copy;     // 1: one copy brings both halves and all atoms of a stage's weight tile (map_b0); 0: one per half and atom
  int half;         // rotary epilogue: pair indices per head (half its width), else 0
  int stages;
  float* scratch;   // [gridDim.x][2][128][BN] fp32 partial tiles
  unsigned* counters;  // one per column tile, zero between launches
  unsigned* status;
};

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// first unit of CTA g when U units are dealt to G CTAs
// (units are counted in 32 bits: a 64-bit division is a subroutine call, which no path of this kernel may contain; the
// host checks that U * G fits)
__device__ __forceinline__ int st_first_unit(int U, int G, int g) { return (int)((unsigned)U * (unsigned)g / (unsigned)G); }
// CTA that owns unit u
__device__ __forceinline__ int st_owner(int U, int G, int u) { return (int)(((unsigned)(u + 1) * (unsigned)G + (unsigned)U - 1u) / (unsigned)U) - 1; }

constexpr int ST_THREADS = 224;
// Every CTA reads the same activations.  Were all to walk K from its start, the whole chip would ask for the same few lines of L2
// at a time; so column tile t starts t * ST_ROT chunks later (and wraps): a LLaDA-shaped pass of 101 rows 4.25 -> 4.16 ms, of 9
// rows 3.72 -> 3.68 (1 to 19 chunks: 4.15 to 4.23, 3.68 to 3.70).  The order depends on the tile alone, so the CTAs that share a
// tile still cover it, and results do not depend on timing.
constexpr int ST_ROT = 4;

// kChains: the rotary epilogue of few rows, whose tiles take K as args.chains slices, one whole tile per CTA: a kernel of its own, as the one without
// them runs with up to 128 rows and was 0.5 to 0.8 % of a pass slower for them.
template <int BN, typename Epi, bool kChains = false>
__global__ void __launch_bounds__(ST_THREADS, 1)
k_gemm_stream(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b0,
              const __grid_constant__ CUtensorMap map_b1, StreamArgs args, Epi epi) {
  extern __shared__ uint8_t smem_raw[];
  constexpr bool kRope = std::is_same<Epi, EpiQKVRope<bf16>>::value;
  if (!kRope) pdl_release();
  constexpr int HALF = BN / 2;
  constexpr int B_HALF_ATOM = HALF * 128;               // bytes of one half-tile atom (64 K elements)
  constexpr int B_ATOM = BN * 128;
  constexpr int ROWS = UM_BM;                             // accumulator rows
  constexpr int SET_COLS = BN;                            // columns of one accumulator set
  constexpr int NBUF = 2;                                 // accumulator sets in tensor memory
  // tensor memory is allocated in powers of two (192-wide tiles use 384 of 512 columns)
  static_assert(!kChains || (kRope && BN == 128), "up to four accumulators of a tile");
  constexpr uint32_t TMEM_COLS = kChains ? 512 : (NBUF * SET_COLS <= 128) ? 128 : (NBUF * SET_COLS <= 256 ? 256 : 512);
  const int A_ATOM = args.a_rows * 128;
  const int AT = args.atoms;
  const int STAGE_BYTES = AT * (A_ATOM + B_ATOM);
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int S = args.stages;
  // (the MMA reads 128 activation rows whatever the box holds: the rest lies in the same stage, whose weight tile is longer)
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)S * STAGE_BYTES);
  // bars[0..S) full, [S..2S) empty, [2S..2S+2) accumulator full, [2S+2..2S+4) accumulator empty
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 4);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  volatile uint32_t* epi_flag = tmem_slot + 2;          // epilogue warps: this CTA finishes the tile
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar_base = smem_u32(bars);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (S + s); };
  auto accf_bar = [&](int b) { return bar_base + 8u * (2 * S + b); };
  auto acce_bar = [&](int b) { return bar_base + 8u * (2 * S + 2 + b); };

  const int G = gridDim.x, g = blockIdx.x;
  const int T = args.n_tiles;
  const int U = T * args.kc;
  // CTA g owns the contiguous units [U g / G, U (g + 1) / G)
  const int u0 = st_first_unit(U, G, g), u1 = st_first_unit(U, G, g + 1);
  const int n_units = (int)(u1 - u0);
  int cl_tile = 0;                   // cluster mode: the tile this CTA contributed a K slice to

  // Position of the producer in the unit space, advanced without divisions (its loop has to keep ahead of the tensor pipe).
  // A tile takes its K chunks in rotated order, starting at chunk rot (see ST_ROT).
  struct Pos {
    int tile, c, rot;
  };
  auto chunk = [&](const Pos& p) { return p.c + p.rot < args.kc ? p.c + p.rot : p.c + p.rot - args.kc; };
  // With several accumulators (chain i takes chunks [kc i / chains, kc (i + 1) / chains) of that order) two neighbouring tiles have the
  // order of the 256-wide tile they make up, and the odd one starts with its second accumulator.
  auto chain_lo = [&](int i) { return args.kc * i / args.chains; };
  auto rot_of = [&](int tile) {
    return (kChains ? (tile >> 1) * ST_ROT + chain_lo(tile & 1) : tile * ST_ROT) % args.kc;
  };
  auto pos_set = [&](Pos& p, int u) {
    p.tile = u / args.kc;
    p.c = u % args.kc;
    p.rot = rot_of(p.tile);
  };
  auto pos_next = [&](Pos& p) {
    if (++p.c == args.kc) { p.c = 0; ++p.tile; p.rot = rot_of(p.tile); }
  };
  // the weight tile of one stage: both halves of every K atom (see umma_map5)
  auto load_weights = [&](const Pos& p, int s) {
    const uint32_t sb = smem_u32(smem + (size_t)s * STAGE_BYTES) + AT * A_ATOM;
    const int j = p.tile * (Epi::kDual ? HALF : BN);
    const int r0 = args.half ? 0 : j, blk = args.half ? j / args.half : 0, a0 = chunk(p) * AT;
    if (args.one_copy) {
      tma_load_5d(sb, &map_b0, r0, blk, 0, a0, full_bar(s));
    } else {
      for (int a = 0; a < AT; ++a) {
        tma_load_5d(sb + a * B_ATOM, &map_b0, r0, blk, 0, a0 + a, full_bar(s));
        tma_load_5d(sb + a * B_ATOM + B_HALF_ATOM, &map_b1, r0, blk, 0, a0 + a, full_bar(s));
      }
    }
  };
  auto load_acts = [&](const Pos& p, int s) {
    tma_load_4d(smem_u32(smem + (size_t)s * STAGE_BYTES), &map_a, 0, 0, chunk(p) * AT, full_bar(s));
  };

  const int n_pre = n_units < S ? n_units : S;      // stages whose weights are requested before the predecessor is done
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf_bar(b), 1);
      mbar_init(acce_bar(b), 4);
    }
    *abort_flag = 0;
    *epi_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  // The weights are never written by any kernel, so the first stages' weight tiles can be requested at once, while a preceding
  // kernel (launched with programmatic serialisation) is still running: the first one here, the others after the set-up's
  // barrier, which nobody is to wait for them at (a full ring's requests take the copy engine 2 us).
  Pos pw;
  pos_set(pw, u0);
  auto request_weights = [&](int s) {
    if (elect_one()) {
      mbar_expect_tx(full_bar(s), STAGE_BYTES);
      load_weights(pw, s);
    }
    __syncwarp();
    pos_next(pw);
  };
  if (warp == 0) {
    __syncwarp();
    if (n_pre > 0) request_weights(0);
  }
  if (threadIdx.x == 64) tma_prefetch_map(&map_a);      // its first use comes right after pdl_wait()
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // barriers and tensor memory are set up; every role waits for the preceding kernel before it reads what that wrote, and before
  // its first bounded wait
  if (warp == 0) {
    // ---------------- TMA producer of the weights: one uninterrupted stream over this CTA's units ----------------
    for (int it = 1; it < n_pre; ++it) request_weights(it);
    pdl_wait();
    int issued = n_pre, s = 0;
    uint32_t ph = 1;
    for (int it = n_pre; it < n_units; ++it) {
      if (!__all_sync(0xffffffffu, mbar_wait(empty_bar(s), ph ^ 1u, abort_flag))) {
        if (lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(args.status, 1u); args.status[1] = 11u; }
        um_let_land();
        break;
      }
      request_weights(s);
      ++issued;
      if (++s == S) { s = 0; ph ^= 1u; }
    }
    // do not leave while copies, these or the activations', may still be landing in this CTA's shared memory
    for (int it = issued > S ? issued - S : 0; it < issued; ++it) {
      if (!__all_sync(0xffffffffu, mbar_wait(full_bar(it % S), (uint32_t)(it / S) & 1u, abort_flag))) {
        um_let_land();
        break;
      }
    }
  } else if (warp == 6) {
    // ---------------- TMA producer of the activations ----------------
    // (the same stages in the same order; they may arrive ahead of the stage's arming: its phase ends with both.  A warp of its
    // own: behind the weights that fill the ring its first request would wait 2 us.)
    pdl_wait();
    if (kRope) pdl_release();        // the attention that follows reads older keys and values ahead of its own wait
    Pos p;
    pos_set(p, u0);
    int s = 0;
    uint32_t ph = 0;
    for (int it = 0; it < n_units; ++it) {
      if (it >= n_pre && !__all_sync(0xffffffffu, mbar_wait(empty_bar(s), ph ^ 1u, abort_flag))) {
        if (lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(args.status, 1u); args.status[1] = 15u; }
        um_let_land();
        break;
      }
      if (elect_one()) load_acts(p, s);
      __syncwarp();
      if (++s == S) { s = 0; ph ^= 1u; }
      pos_next(p);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (the whole warp waits, one elected thread issues) ----------------
    {
      pdl_wait();
      constexpr uint32_t idesc = make_idesc(BN);
      int seg = 0;
      bool ok = true, ready = false;           // ready: stage s has been seen full
      int s = 0;
      uint32_t ph = 0;
      for (int u = u0; u < u1 && ok;) {
        const int vt = (int)(u / args.kc);
        const int seg_end = min(u1, (vt + 1) * args.kc);
        const int buf = seg % NBUF, use = seg / NBUF;
        // wait until the epilogue has drained this accumulator set (its previous use was segment seg - NBUF)
        if (use >= 1) ok = __all_sync(0xffffffffu, mbar_wait(acce_bar(buf), (uint32_t)(use - 1) & 1u, abort_flag));
        if (!ok) {
          if (lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(args.status, 1u); args.status[1] = 12u; }
          break;
        }
        tc_fence_after();
        uint32_t d_tmem = tmem_base + (uint32_t)(buf * SET_COLS);
        uint32_t acc = 0;                               // 0: the next MMA overwrites the accumulator
        int chain = 0, next_acc = seg_end;              // the first unit of the next accumulator
        if (kChains) {
          chain = (vt & 1) % args.chains;
          d_tmem += (uint32_t)(chain * BN);
          next_acc = u + chain_lo(chain + 1) - chain_lo(chain);
        }
        for (; u < seg_end; ++u) {
          if (kChains && u == next_acc) {
            if (++chain == args.chains) chain = 0;
            d_tmem = tmem_base + (uint32_t)(chain * BN);
            acc = 0;
            next_acc = u + chain_lo(chain + 1) - chain_lo(chain);
          }
          if (!ready) ok = __all_sync(0xffffffffu, mbar_wait(full_bar(s), ph, abort_flag));
          if (!ok) {
            if (lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(args.status, 1u); args.status[1] = 13u; }
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + (size_t)s * STAGE_BYTES);
          const uint32_t sb = sa + AT * A_ATOM;
          int s2 = s + 1;
          uint32_t ph2 = ph;
          if (s2 == S) { s2 = 0; ph2 ^= 1u; }
          if (AT == 2) {
            if (elect_one()) {
              const uint64_t da = make_smem_desc(sa), db = make_smem_desc(sb);
#pragma unroll
              for (int k = 0; k < 4; ++k) tc_mma_f16(d_tmem, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc, acc | (uint32_t)k);
            }
            __syncwarp();
            acc = 1;
          }
          // the next stage is looked at between this one's MMAs, while the tensor pipe still has work
          ready = __all_sync(0xffffffffu, mbar_test(full_bar(s2), ph2));
          if (elect_one()) {
            const uint64_t da = make_smem_desc(sa + (AT - 1) * A_ATOM), db = make_smem_desc(sb + (AT - 1) * B_ATOM);
#pragma unroll
            for (int k = 0; k < 4; ++k) tc_mma_f16(d_tmem, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc, acc | (uint32_t)k);
            tc_commit(empty_bar(s));
            if (u == seg_end - 1) tc_commit(accf_bar(buf));
          }
          __syncwarp();
          acc = 1;
          s = s2;
          ph = ph2;
        }
        ++seg;
      }
    }
  } else {
    // ---------------- epilogue (warps 2..5) ----------------
    pdl_wait();
    const int q = warp & 3;
    const int r_in = q * 32 + lane;                       // accumulator lane this thread reads
    constexpr int CH = Epi::kDual ? HALF : BN;            // pair indices (dual) or columns (plain) per tile
    int seg = 0;
    bool ok = true;
    for (int u = u0; u < u1 && ok; ++seg) {
      const int vt = (int)(u / args.kc);
      const int tile = vt;
      const int tile_u0 = vt * args.kc;
      const int seg_end = min(u1, tile_u0 + args.kc);
      const bool whole = kChains || ((u == tile_u0) && (seg_end == tile_u0 + args.kc));
      const int buf = seg % NBUF, use = seg / NBUF;
      const int j0 = tile * CH;
      // what the first chunk's epilogue reads is fetched while the MMAs run (see EpiPre)
      EpiPre<Epi> preA, preB;
      if constexpr (!Epi::kReduce) {
        if (whole && r_in < args.M && j0 < args.n_pairs) preA.load(epi, r_in, j0);
      }
      if (!__all_sync(0xffffffffu, mbar_wait(accf_bar(buf), (uint32_t)use & 1u, abort_flag))) {
        if (lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(args.status, 1u); args.status[1] = 14u; }
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * SET_COLS);
      if (whole) {
        // the accumulator is complete in tensor memory: each thread owns one row
        {
          const int m = r_in;
          Top2 red = top2_empty();
          // one chunk of 16 columns (or pairs) at a time; the next chunk's tensor-memory loads are in flight while this
          // one is converted and stored
          auto fetch = [&](int c, EpiPre<Epi>& pre) {
            if constexpr (!Epi::kReduce) {
              if (m < args.M && c < CH && j0 + c < args.n_pairs) pre.load(epi, m, j0 + c);
            }
          };
          auto consume = [&](int c, float (&a0)[16], float (&a1)[16], const EpiPre<Epi>& pre) {
            if constexpr (Epi::kReduce) {
              top2_push16(red, a0, j0 + c, epi);
            } else {
              if (m < args.M && j0 + c < args.n_pairs) epi16(epi, m, j0 + c, a0, a1, pre);
            }
            __syncwarp();
          };
          auto request = [&](int c, float (&a0)[16], float (&a1)[16]) {
            tc_ld16_nowait(t_row + c, a0);
            if (Epi::kDual) tc_ld16_nowait(t_row + HALF + c, a1);
          };
          if constexpr (kRope) {
            // (the table entries of two chunks take the registers a second set of accumulator values would)
            float p0[16], p1[16];
#pragma unroll 1
            for (int c = 0; c < CH; c += 16) {
              request(c, p0, p1);
              fetch(c + 16, preB);
              tc_wait_ld();
              tc_pin16(p0);
              tc_pin16(p1);
              if constexpr (kChains) {
#pragma unroll 1
                for (int x = 1; x < args.chains; ++x) {            // in K order
                  float v[16];
                  tc_ld16(t_row + (uint32_t)(x * BN + c), v);
#pragma unroll
                  for (int i = 0; i < 16; ++i) p0[i] += v[i];
                  tc_ld16(t_row + (uint32_t)(x * BN + HALF + c), v);
#pragma unroll
                  for (int i = 0; i < 16; ++i) p1[i] += v[i];
                }
              }
              consume(c, p0, p1, preA);
              preA = preB;
            }
          } else {
          float p0[16], p1[16], q0[16], q1[16];
          request(0, p0, p1);
#pragma unroll 1
          for (int c = 0; c < CH; c += 32) {
            tc_wait_ld();
            tc_pin16(p0);
            if (Epi::kDual) tc_pin16(p1);
            if (c + 16 < CH) request(c + 16, q0, q1);
            fetch(c + 16, preB);
            consume(c, p0, p1, preA);
            if (c + 16 < CH) {                     // CH is a multiple of 16, not always of 32 (48 pairs per tile)
              tc_wait_ld();
              tc_pin16(q0);
              if (Epi::kDual) tc_pin16(q1);
              if (c + 32 < CH) request(c + 32, p0, p1);
              fetch(c + 32, preA);
              consume(c + 16, q0, q1, preB);
            }
          }
          }
          if constexpr (Epi::kReduce) {
            if (m < args.M) epi.part[(size_t)m * epi.n_tiles + tile] = red;
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce_bar(buf));
      } else {
        // publish this CTA's partial tile, then count its chunks in; the CTA that completes the count finishes the tile.
        // Partial tile layout: [16-column chunk][quarter][row][4 floats], so that the lanes of a warp (consecutive
        // rows) write and read consecutive 16-byte pieces.
        // With clusters the partial tile goes to this CTA's own shared memory (the pipeline stages are idle by now) and
        // is reduced after the role loops; without, to the global scratch slot of this CTA.
        if (args.exchange) {
          // Exchange between the two CTAs of a pair: each finishes half of the tile's 16-column chunks, so each
          // publishes only the half its peer will finish and keeps its own half in tensor memory (see below).
          constexpr int P = Epi::kDual ? 2 : 1;
          const int rank = (int)cluster_ctarank();
          const int p_lo = (CH / 16) * (1 - rank) / 2, p_hi = (CH / 16) * (2 - rank) / 2;     // the peer's chunks
          float4* slot = reinterpret_cast<float4*>(smem);
          if (q * 32 < args.M) {                          // else none of this warp's rows exists
#pragma unroll 1
            for (int ch = p_lo; ch < p_hi; ++ch) {
#pragma unroll
              for (int p = 0; p < P; ++p) {
                float v[16];
                __syncwarp();
                tc_ld16(t_row + p * HALF + ch * 16, v);
                if (r_in < args.M) {
#pragma unroll
                  for (int i = 0; i < 4; ++i)
                    slot[(size_t)(((ch - p_lo) * P + p) * 4 + i) * ROWS + r_in] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                }
              }
            }
          }
          cl_tile = tile;
          u = seg_end;
          continue;
        }
        float4* slot_base = args.cluster > 1
                                ? reinterpret_cast<float4*>(smem)
                                : reinterpret_cast<float4*>(args.scratch + (size_t)(g * 2 + (seg == 0 ? 0 : 1)) * ROWS * BN);
        if (q * 32 < args.M) {                            // else none of this warp's rows exists
#pragma unroll 1
          for (int c = 0; c < BN; c += 16) {
            float v[16];
            __syncwarp();
            tc_ld16(t_row + c, v);
            if (r_in < args.M) {
#pragma unroll
              for (int i = 0; i < 4; ++i)
                slot_base[(size_t)((c >> 4) * 4 + i) * ROWS + r_in] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
          }
        }
        // the accumulator set is free as soon as every warp has read it
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce_bar(buf));
        if (args.cluster > 1) {          // reduced after the cluster barrier below
          cl_tile = tile;
          u = seg_end;
          continue;
        }
        __threadfence();
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (threadIdx.x == 64) {
          const unsigned add = (unsigned)(seg_end - u);
          const unsigned old = atomicAdd(args.counters + tile, add);
          const bool last = (old + add == (unsigned)args.kc);
          if (last) args.counters[tile] = 0;          // ready for the next launch
          *epi_flag = last ? 1u : 0u;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (*epi_flag != 0) {
          __threadfence();
          const int g_lo = st_owner(U, G, tile_u0), g_hi = st_owner(U, G, tile_u0 + args.kc - 1);
          // The tile is the sum of the contributors' partial tiles.  Work items are (row, 16-column chunk), dealt over
          // the 128 epilogue threads so that a tile with few rows still uses all of them, and every item issues the
          // loads of several contributors before it adds them (in CTA order: deterministic).
          constexpr int NCH = CH / 16;                 // chunks per row
          constexpr int RPP = 128 / NCH;               // rows per pass
          const int et = threadIdx.x - 64;
          // plain epilogues: consecutive lanes take consecutive rows (coalesced reads of the partials); the reducing
          // epilogue keeps a row's chunks in neighbouring lanes so that they can be merged with shuffles
          const int ch = Epi::kReduce ? et % NCH : et / RPP, c = ch * 16;
          const int rows_here = args.M;
          for (int mm0 = 0; mm0 < rows_here; mm0 += RPP) {
            const int mm = mm0 + (Epi::kReduce ? et / NCH : et % RPP);
            const bool valid = mm < rows_here;
            float a0[16], a1[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) { a0[i] = 0.f; a1[i] = 0.f; }
            if (valid) {
              constexpr int GB = Epi::kDual ? 2 : 4;
              for (int gb = g_lo; gb <= g_hi; gb += GB) {
                float4 t0[GB][4], t1[GB][4];
#pragma unroll
                for (int x = 0; x < GB; ++x) {
                  const int gg = gb + x;
                  if (gg <= g_hi) {
                    // contributor gg's segment of this tile is its first one iff its share starts inside the tile
                    const int slot = (st_first_unit(U, G, gg) >= tile_u0) ? 0 : 1;
                    const float4* base = reinterpret_cast<const float4*>(args.scratch + (size_t)(gg * 2 + slot) * ROWS * BN) + mm;
                    const float4* p0 = base + (size_t)(c >> 4) * 4 * ROWS;
#pragma unroll
                    for (int i = 0; i < 4; ++i) t0[x][i] = __ldcg(p0 + (size_t)i * ROWS);
                    if (Epi::kDual) {
                      const float4* p1 = base + (size_t)((HALF + c) >> 4) * 4 * ROWS;
#pragma unroll
                      for (int i = 0; i < 4; ++i) t1[x][i] = __ldcg(p1 + (size_t)i * ROWS);
                    }
                  }
                }
#pragma unroll
                for (int x = 0; x < GB; ++x) {
                  if (gb + x <= g_hi) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                      a0[4 * i] += t0[x][i].x; a0[4 * i + 1] += t0[x][i].y; a0[4 * i + 2] += t0[x][i].z; a0[4 * i + 3] += t0[x][i].w;
                      if (Epi::kDual) {
                        a1[4 * i] += t1[x][i].x; a1[4 * i + 1] += t1[x][i].y; a1[4 * i + 2] += t1[x][i].z; a1[4 * i + 3] += t1[x][i].w;
                      }
                    }
                  }
                }
              }
            }
            if constexpr (Epi::kReduce) {
              Top2 red = top2_empty();
              if (valid) top2_push16(red, a0, j0 + c, epi);
#pragma unroll
              for (int o = 1; o < NCH; o <<= 1) red = top2_merge(red, top2_shfl_xor(red, o));
              if (valid && ch == 0) epi.part[(size_t)mm * epi.n_tiles + tile] = red;
            } else {
              if (valid && j0 + c < args.n_pairs) epi16(epi, mm, j0 + c, a0, a1);
            }
          }
        }
      }
      u = seg_end;
    }
  }
  if (!kChains && args.exchange) {
    // Pair exchange: after the barrier each CTA adds, for its own half of the chunks, its accumulator (still in tensor
    // memory) and the peer's published piece, and runs the fused epilogue.  One row per thread, as in the plain epilogue;
    // the next chunk's piece and what its epilogue reads are requested before the current one is finished.
    if constexpr (!Epi::kReduce) {
      constexpr int CH = Epi::kDual ? HALF : BN;
      constexpr int P = Epi::kDual ? 2 : 1;
      const int rank = (int)cluster_ctarank();
      const int o_lo = (CH / 16) * rank / 2, n_ch = (CH / 16) * (rank + 1) / 2 - o_lo;        // this CTA's chunks
      const int q = warp & 3, r_in = q * 32 + lane;
      const bool mine = warp >= 2 && warp <= 5 && n_units > 0;
      const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16);
      const uint32_t peer = cluster_map(smem_u32(smem), (unsigned)(rank ^ 1));
      const int j0 = cl_tile * CH;
      auto live = [&](int it) { return it < n_ch && r_in < args.M && j0 + (o_lo + it) * 16 < args.n_pairs; };
      auto fetch = [&](int it, EpiPre<Epi>& pre) {
        if (live(it)) pre.load(epi, r_in, j0 + (o_lo + it) * 16);
      };
      auto request = [&](int it, float4 (&t0)[4], float4 (&t1)[4]) {
        if (live(it)) {
#pragma unroll
          for (int i = 0; i < 4; ++i) t0[i] = ld_cluster_f4(peer + (uint32_t)(((it * P * 4 + i) * ROWS + r_in) * 16));
          if (Epi::kDual) {
#pragma unroll
            for (int i = 0; i < 4; ++i) t1[i] = ld_cluster_f4(peer + (uint32_t)((((it * P + 1) * 4 + i) * ROWS + r_in) * 16));
          }
        }
      };
      auto finish = [&](int it, const float4 (&t0)[4], const float4 (&t1)[4], const EpiPre<Epi>& pre) {
        const int ch = o_lo + it;
        float a0[16], a1[16];
        __syncwarp();
        tc_ld16(t_row + ch * 16, a0);
        if (Epi::kDual) tc_ld16(t_row + HALF + ch * 16, a1);
        if (live(it)) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            a0[4 * i] += t0[i].x; a0[4 * i + 1] += t0[i].y; a0[4 * i + 2] += t0[i].z; a0[4 * i + 3] += t0[i].w;
            if (Epi::kDual) {
              a1[4 * i] += t1[i].x; a1[4 * i + 1] += t1[i].y; a1[4 * i + 2] += t1[i].z; a1[4 * i + 3] += t1[i].w;
            }
          }
          epi16(epi, r_in, j0 + ch * 16, a0, a1, pre);
        }
      };
      EpiPre<Epi> preA, preB;
      if (mine) fetch(0, preA);
      cluster_sync();
      // a warp whose rows do not exist has nothing to finish
      const int n_it = (mine && q * 32 < args.M) ? n_ch : 0;
      if (n_it > 0) {
        tc_fence_after();
        float4 a0[4], a1[4], b0[4], b1[4];
        request(0, a0, a1);
        if constexpr (kRope) {              // (registers: one piece at a time)
#pragma unroll 1
          for (int it = 0; it < n_it; ++it) {
            finish(it, a0, a1, preA);
            request(it + 1, a0, a1);
            fetch(it + 1, preA);
          }
        } else {
#pragma unroll 1
        for (int it = 0; it < n_it; it += 2) {
          request(it + 1, b0, b1);
          fetch(it + 1, preB);
          finish(it, a0, a1, preA);
          if (it + 1 < n_it) {
            request(it + 2, a0, a1);
            fetch(it + 2, preA);
            finish(it + 1, b0, b1, preB);
          }
        }
        }
      }
    } else {
      cluster_sync();
    }
    cluster_sync();      // nobody leaves while its peer may still read its shared memory
  } else if (!kChains && args.cluster > 1) {
    // Split-K reduction inside the cluster: every CTA's partial tile sits in its shared memory; after the barrier CTA
    // rank r sums, for its share of the 16-column chunks, the partials of all ranks in rank order (= K order, so the
    // result does not depend on timing) straight from their shared memory, and runs the fused epilogue on them.
    // Every thread of every CTA reaches both barriers (no early exits above), so they cannot hang.
    const int C = args.cluster;
    {
      if constexpr (Epi::kReduce) {
        cluster_sync();
      } else {
        constexpr int CH = Epi::kDual ? HALF : BN;
        constexpr int NCH = CH / 16;
        const unsigned rank = cluster_ctarank();
        const int ch_lo = NCH * (int)rank / C, ch_hi = NCH * ((int)rank + 1) / C;
        const int rows_here = args.M;
        const int n_items = (warp >= 2 && warp <= 5 && n_units > 0) ? rows_here * (ch_hi - ch_lo) : 0;
        const int j0 = cl_tile * CH;
        // what an item's epilogue reads is fetched before the barrier, then one item ahead
        EpiPre<Epi> pre, next;
        auto fetch = [&](int idx, EpiPre<Epi>& p) {
          if (idx >= 0 && idx < n_items) {               // (threads of the first two warps pass negative indices)
            const int c = (ch_lo + idx / rows_here) * 16;
            if (j0 + c < args.n_pairs) p.load(epi, idx % rows_here, j0 + c);
          }
        };
        fetch((int)threadIdx.x - 64, pre);
        cluster_sync();
        if (n_items > 0) {
          const uint32_t base = smem_u32(smem);
          for (int idx = threadIdx.x - 64; idx < n_items; idx += 128) {
            const int mm = idx % rows_here, ch = ch_lo + idx / rows_here, c = ch * 16;
            if (!kRope) fetch(idx + 128, next);          // (registers: a rotary item's table entries follow the item)
            float a0[16], a1[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) { a0[i] = 0.f; a1[i] = 0.f; }
            const uint32_t off0 = (uint32_t)(((c >> 4) * 4 * ROWS + mm) * 16);
            const uint32_t off1 = (uint32_t)((((HALF + c) >> 4) * 4 * ROWS + mm) * 16);
            // several ranks' pieces are requested before any is added (the loads are independent; the sum stays in rank
            // order): four, or two where an item is a pair of chunks
            constexpr int PB = Epi::kDual ? 2 : 4;
            for (int pb = 0; pb < C; pb += PB) {
              float4 t0[PB][4], t1[PB][4];
#pragma unroll
              for (int x = 0; x < PB; ++x) {
                if (pb + x < C) {
                  const uint32_t peer = cluster_map(base, (unsigned)(pb + x));
#pragma unroll
                  for (int i = 0; i < 4; ++i) t0[x][i] = ld_cluster_f4(peer + off0 + (uint32_t)(i * ROWS * 16));
                  if (Epi::kDual) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) t1[x][i] = ld_cluster_f4(peer + off1 + (uint32_t)(i * ROWS * 16));
                  }
                }
              }
#pragma unroll
              for (int x = 0; x < PB; ++x) {
                if (pb + x < C) {
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    a0[4 * i] += t0[x][i].x; a0[4 * i + 1] += t0[x][i].y; a0[4 * i + 2] += t0[x][i].z; a0[4 * i + 3] += t0[x][i].w;
                    if (Epi::kDual) {
                      a1[4 * i] += t1[x][i].x; a1[4 * i + 1] += t1[x][i].y; a1[4 * i + 2] += t1[x][i].z; a1[4 * i + 3] += t1[x][i].w;
                    }
                  }
                }
              }
            }
            if (j0 + c < args.n_pairs) epi16(epi, mm, j0 + c, a0, a1, pre);
            if (kRope) fetch(idx + 128, pre);
            else pre = next;
          }
        }
      }
      cluster_sync();      // nobody leaves while a peer may still read its shared memory
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// ---- host side ------------------------------------------------------------------------------------------------
// Scratch the streaming kernel needs for a grid of n_ctas CTAs of tile width bn.
inline size_t stream_scratch_bytes(int n_ctas, int bn) { return (size_t)n_ctas * 2 * UM_BM * bn * sizeof(float); }

// Number of CTAs.  Dealing the units evenly over all SMs balances the weight stream perfectly but splits almost every
// tile between two CTAs, which costs a partial tile written and read back per split (M x BN x 4 bytes each way).
// With at most as many tiles as SMs, a grid that is a multiple of the tile count splits each tile into equal K slices
// instead (no split at all when there are more than half as many tiles as SMs).  Measured on the LLaDA layer shapes
// the second choice is as fast or faster at every row count from 2 to 128, so it is the default.
// K slices per tile when the tiles are fewer than the SMs.  With clusters on, the slices of a tile form one cluster of 2
// to 8 CTAs, and a launch never asks for more clusters than can be resident at once: the GPC layout fits 74 / 45 / 33 /
// 26 / 22 / 15 / 15 clusters of 2 ... 8 one-per-SM CTAs, so e.g. 48 clusters of 3 or 16 of 8 would run as two waves
// (measured: 40 % and 100 % slower than the next smaller split).
// With a short K (at most 512) a slice would be a stage or two, and the reduction costs more than it saves, except where the
// epilogue reads its output's old value (see no_split): 64 x 2 x 1024 SwiGLU 9.7 -> 7.2 us, 100 x 1024 6.8 -> 5.2, 64 x 4096
// 6.2 -> 4.9 unsplit, but a residual update of 100 x 512 7.5 -> 8.0; from K = 1024 on the split wins (64 x 512 6.8, 8.9 without).
// With few rows a dual epilogue, whose tiles are 256 wide, loses by it: SwiGLU of 1024 pairs (K 512) at 1 / 9 / 16 / 24 rows 6.3 / 6.7 / 6.9 /
// 7.1 us split, 7.4 / 7.4 / 7.3 / 7.3 whole, eight layers (d 512) at 3 rows 332 and 355.  It stays whole at every row count: a sum whose
// order changed with the rows moved near-tied predictions of such a model (one token in five of sixty decodes).
// The head, with few tiles and a short K, comes here with at most 8 rows (umma_head_shape) and keeps the split: 4 rows of 4096 ids
// 15.1 -> 12.9 us, and the shorter sums are more exact.
template <typename Epi>
bool stream_no_split(int K) { return K <= 512 && !Epi::kReduce && !std::is_same<Epi, EpiResidual<bf16>>::value; }
inline int stream_splits(const UmmaState& st, long n_tiles, bool no_split) {
  int splits = n_tiles <= st.n_sm ? (int)(st.n_sm / n_tiles) : 0;
  if (no_split && splits > 1) return 1;
  if (st.stream_cluster && splits > 1) {
    int c = splits < 8 ? splits : 8;
    while (c > 1 && n_tiles > st.max_clusters[c]) --c;
    splits = c;
  }
  return splits;
}

inline int stream_grid(const UmmaState& st, int n_tiles, int bn, bool no_split) {
  // (a forced count: as many as the scratch holds partial tiles for)
  if (st.target_ctas > 0) return std::min(st.target_ctas, (int)(st.scratch_bytes / stream_scratch_bytes(1, bn)));
  const int splits = stream_splits(st, n_tiles, no_split);
  return (st.stream_even || splits == 0) ? st.n_sm : n_tiles * splits;
}

// Stage shape for an activation box of a_rows rows and tile width bn: two K atoms per stage when at least
// stream_min_stages2 such stages fit.
struct StreamShape { int a_rows, atoms, stages, stage_bytes, aux; };
inline StreamShape stream_shape(const UmmaState& st, int M, int bn, int K) {
  StreamShape sh;
  sh.a_rows = (M + 7) / 8 * 8;
  sh.aux = 1024 + 8 * (2 * ST_MAX_STAGES + 4) + 16;
  const int atom = sh.a_rows * 128 + bn * 128;
  sh.atoms = (K % 128 == 0 && (st.max_smem - sh.aux) / (2 * atom) >= st.stream_min_stages2) ? 2 : 1;
  if (st.stream_atoms == 1 || (st.stream_atoms == 2 && K % 128 == 0)) sh.atoms = st.stream_atoms;
  sh.stage_bytes = sh.atoms * atom;
  sh.stages = (st.max_smem - sh.aux) / sh.stage_bytes;
  if (sh.stages > ST_MAX_STAGES) sh.stages = ST_MAX_STAGES;
  if (sh.stages > st.max_stages) sh.stages = st.max_stages;
  return sh;
}

// Most bytes between the two halves (gate and up) of a weight tile that one copy brings.  A tensor map takes strides up to 2^40, but a box
// that spans more than a gigabyte read elsewhere: with the tensors 1.18 GB apart (64 pairs, K 512) a launch ended in an illegal memory
// access, at 0.83 GB and below it does not.  Halves further apart come by a copy each: with those 30 cases up to 4.4 GB apart are right.
constexpr size_t ST_MAX_SPAN = (size_t)1 << 29;

// Asks the runtime how many clusters of 2 ... 8 CTAs of the streaming kernel (one CTA per SM) can be resident at once.
inline void stream_query_clusters(UmmaState& st) {
  auto kern = k_gemm_stream<128, EpiStore<bf16>>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, st.max_smem) != cudaSuccess) return;
  st.max_clusters[1] = st.n_sm;
  for (int c = 2; c <= 8; ++c) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * c * st.n_sm);
    cfg.blockDim = dim3(ST_THREADS);
    cfg.dynamicSmemBytes = (size_t)st.max_smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)c;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0) st.max_clusters[c] = n;
  }
  cudaGetLastError();
}

template <int BN, typename Epi>
int stream_launch(UmmaState& st, cudaStream_t stream, const bf16* A, const bf16* W0, const bf16* W1, int M, int NP, int K,
                  int n_rows_w, const Epi& epi, unsigned* status) {
  const StreamShape sh = stream_shape(st, M, BN, K);
  if (sh.stages < 2) { st.err = "not enough shared memory for the streaming GEMM"; return -2; }
  const size_t smem = (size_t)sh.stages * sh.stage_bytes + sh.aux;
  const CUtensorMap* ma = umma_map4(st, A, M, M, 1, K, sh.a_rows, 1, sh.atoms);
  if (!ma) return -4;
  WeightView v{W0, n_rows_w, 1, n_rows_w, 1, 0, BN, 1};
  int one_copy = 1, rot_half = 0;
  Epi e2 = epi;
  if constexpr (std::is_same<Epi, EpiQKVRope<bf16>>::value) {
    rot_half = epi.half;
    v = WeightView{W0, rot_half, n_rows_w / (2 * rot_half), 2 * rot_half, 2, (size_t)rot_half * K * 2, rot_half, BN / 2 / rot_half};
  } else if constexpr (Epi::kDual) {
    // gate and up are two tensors: the halves' distance is that of the tensors (either may come first)
    const bool flip = (uintptr_t)W1 < (uintptr_t)W0;
    const size_t dist = flip ? (const char*)W0 - (const char*)W1 : (const char*)W1 - (const char*)W0;
    v = WeightView{flip ? W1 : W0, n_rows_w, 1, n_rows_w, 2, dist, BN / 2, 1};
    if (dist == 0 || dist >= ST_MAX_SPAN || (dist & 15) || st.stream_split_copies) { one_copy = 0; v.base = W0; v.halves = 1; }
    else if (flip) e2.flip = 1;
  }
  const CUtensorMap* mb0 = umma_map5(st, v, K, one_copy ? sh.atoms : 1);
  if (!mb0) return -4;
  const CUtensorMap mb0v = *mb0;
  CUtensorMap mb1v = mb0v;
  if (!one_copy) {
    v.base = W1;
    const CUtensorMap* mb1 = umma_map5(st, v, K, 1);
    if (!mb1) return -4;
    mb1v = *mb1;
  }
  const int per_tile = Epi::kDual ? BN / 2 : BN;
  const int n_tiles = (NP + per_tile - 1) / per_tile;
  const int kc = K / (sh.atoms * UM_BK);
  const long T = n_tiles;
  int grid = stream_grid(st, (int)T, BN, stream_no_split<Epi>(K));
  if (grid > T * kc) grid = (int)(T * kc);
  if ((double)T * kc * (grid + 1) >= 4.0e9) { st.err = "too many work units for the streaming GEMM"; return -9; }   // 32-bit unit arithmetic
  // K slices of one tile on the CTAs of one cluster: the reduction then stays on chip
  int cluster = 0, exchange = 0;
  if (!Epi::kReduce && st.stream_cluster && grid % T == 0) {
    const int splits = (int)(grid / T);
    if (splits >= 2 && splits <= 8 && kc >= splits && (size_t)sh.stages * sh.stage_bytes >= (size_t)UM_BM * BN * sizeof(float)) {
      cluster = splits;
      // (a few rows: their items are better dealt over all epilogue threads than kept by the warp that owns the rows)
      exchange = (splits == 2 && st.stream_exchange && M >= st.stream_exchange_rows) ? 1 : 0;
    }
  }
  // rotary tiles of few rows in place of 256-wide ones (see umma_gemm): as many accumulators as those would have K slices
  int chains = 0;
  if constexpr (std::is_same<Epi, EpiQKVRope<bf16>>::value && BN == 128) {
    if (M <= 32 && grid == T && st.stream_bn == 0)
      chains = std::max(1, std::min(stream_splits(st, (T + 1) / 2, stream_no_split<Epi>(K)), std::min(4, kc)));
  }
  StreamArgs args{M, NP, n_tiles, cluster, exchange, kc, chains, sh.a_rows, sh.atoms, one_copy, rot_half, sh.stages, st.scratch, st.counters, status};
  auto kern = k_gemm_stream<BN, Epi>;
  if constexpr (std::is_same<Epi, EpiQKVRope<bf16>>::value && BN == 128) {
    if (chains > 0) kern = k_gemm_stream<BN, Epi, true>;
  }
  const cudaError_t smem_rc = umma_raise_smem(st, kern);
  if (smem_rc != cudaSuccess) { st.err = cudaGetErrorString(smem_rc); return -3; }
  cudaError_t e = launch_k(st.pdl, kern, dim3(grid), dim3(ST_THREADS), smem, stream, cluster, *ma, mb0v,
                           mb1v, args, e2);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) { st.err = cudaGetErrorString(e); return -5; }
  return 0;
}

// Whether the streaming kernel can take the problem with tiles of bn columns (scratch or counters too small for a split grid,
// too little shared memory).
template <typename Epi>
bool stream_can(const UmmaState& st, int M, int NP, int K, int bn) {
  const long T = (NP + (Epi::kDual ? bn / 2 : bn) - 1) / (Epi::kDual ? bn / 2 : bn);
  if (st.scratch == nullptr || T > st.n_counters || stream_scratch_bytes(stream_grid(st, (int)T, bn, stream_no_split<Epi>(K)), bn) > st.scratch_bytes)
    return false;
  return stream_shape(st, M, bn, K).stages >= 2;
}

}  // namespace lsp
