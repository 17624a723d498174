// Suffix-over-prefix attention of large passes on the 5th-generation tensor cores (tcgen05 + TMEM), head_dim 128, bf16: the contract of
// attention_umma.cuh, whose kernel takes the passes with few CTAs.
//
// Measured against that kernel, passes in ms: 16 x 515 rows over 2100 keys (32 heads) 105.1 -> 103.0; 8 x 154 over 560 18.8 -> 18.5;
// 8 x 205 over 900 (28 heads, 4 KV) 27.7 -> 27.5; 4 x 1024 over 1024 no difference (46.7, 46.6).
// What bounds that kernel with many key tiles is shared memory: per 128 x 128 score tile it writes 64 KB of keys and values and 32 KB of
// softmax weights, and its MMAs read 128 KB: about 1800 of the 2470 cycles a tile takes.  Here
//   * a CTA owns TWO row tiles of 128 (position, head of the group) rows of one (sequence, KV head), which share every K / V tile: half
//     the bytes written per score tile;
//   * each row tile has a softmax group of 128 threads of its own (one row each) and its own accumulator, so nothing is merged at the
//     end; while one group computes, the tensor pipe works for the other;
//   * the weights P go to tensor memory, over the scores they were computed from, and are the A operand of P V from there: neither
//     their store nor the MMAs' reads of them touch shared memory.
// One warp issues all MMAs.  They execute in the order of issue, so P V of a tile and Q K^T of the next one, which writes over P, follow
// each other without a wait.  (PTX states that order for MMAs into one accumulator; between two the kernel rests on the one tensor pipe of
// an SM, as the published attention kernels for this chip that keep P over S do.  A wait in between would put another 530 cycles into the
// chain of about 4000 that a tile takes.)  A commit covers all that was issued before it, so scores that have arrived tell the softmax
// group that its previous P V is complete.
// The running maximum is raised lazily, as in attention_umma.cuh, from the fifth tile on; in the first four it follows the scores (to a
// quarter), and the row sum adds the weights as they were rounded.  Here a row has one maximum where that kernel has two: only the
// weight of a key that was the maximum is 1 and without rounding error, and the sum of the rounded weights takes out what their errors
// share.  Error against 64 bits relative to that kernel's, 500 to 4300 keys, scores of standard deviation 0.3 / 1 / 4: fp32 sum and all
// tiles lazy 1.003 / 1.022 / 1.07 at worst; now 1.001 / 0.998 / 0.92.  With two key tiles that kernel's two maxima are all there are
// (1.015), so it takes those passes.  The launch of 16 x 515 rows over 2100 keys alone 458 -> 494 us (that kernel 464); in passes, which
// run at the power limit, it stays the faster one: see above.  (O gathers all key tiles in one accumulator where that kernel has two: the
// bias of the tensor core's truncation is 1.6e-5 of an output at 4300 keys of one sign, 0.9e-5 there, under a rounding to bf16 of 1.4e-3.)
// Warps 0..3 and 4..7 = softmax groups 0 and 1; warps 8 and 11 = TMA producers of the K and the V tiles, warp 9 = TMEM allocator and MMA
// issuer.  Every wait is bounded; on expiry the kernel records (code, site), drains and returns.
#pragma once
#include "attention_umma.cuh"

namespace lsp {

constexpr int AR_SMEM = 1024 + 2 * AU_TILE /*Q*/ + 2 * 2 * AU_TILE /*K, V stages*/ + 256 /*barriers, flags*/;

__device__ __forceinline__ void tc_mma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_st16u(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]),
        "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}

// grid = (ceil(max rows per sequence * group / 256), n_kv_heads, batch)
__global__ void __launch_bounds__(AU_THREADS, 1)
k_attn_rows(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_ck,
            const __grid_constant__ CUtensorMap map_cv, const __grid_constant__ CUtensorMap map_sk,
            const __grid_constant__ CUtensorMap map_sv, bf16* __restrict__ out, StepDesc sd, int n_heads, int n_kv_heads, int max_len,
            float scale_log2, int inplace, int early, unsigned* status) {
  constexpr int DH = 128;
  extern __shared__ uint8_t smem_raw[];
  pdl_release();
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* Qs = smem;                                   // Q of row tile w at Qs + w * AU_TILE
  uint8_t* KVs = smem + 2 * AU_TILE;                    // stage s: K at s * 2 * AU_TILE, V right behind it
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + 6 * AU_TILE);
  // bars: per stage 0 k_full; 2 k_empty; 4 v_full; 6 v_empty; per group 8 s_full; 10 p_ready; 12 done; 14 q_ready
  constexpr int B_KF = 0, B_KE = 2, B_VF = 4, B_VE = 6, B_SF = 8, B_PR = 10, B_PD = 12, B_Q = 14;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 16);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  const uint32_t bb = smem_u32(bars);
  auto bar = [&](int i) { return bb + 8u * i; };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.z, kvh = blockIdx.y;
  const int G = n_heads / n_kv_heads;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 15; ++i) mbar_init(bar(i), (i >= B_PR && i < B_PD) ? 4 : 1);      // p_ready: four warps arrive
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  // tile rows that stand for no position (G does not divide 128): zeros, so that every accumulator row is finite
  for (int i = (AU_BM / G) * G * 8 + (int)threadIdx.x; i < AU_BM * 8; i += AU_THREADS) {
    const uint32_t off = (uint32_t)((i >> 6) * 1024 + ((i >> 3) & 7) * 128 + (i & 7) * 16);
#pragma unroll
    for (int x = 0; x < 4; ++x) *reinterpret_cast<uint4*>(Qs + x * AU_ATOM + off) = make_uint4(0u, 0u, 0u, 0u);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == AU_W_TMA && lane == 0) {
    tma_prefetch_map(&map_q);
    tma_prefetch_map(&map_ck);
    tma_prefetch_map(&map_sk);
  }
  if (warp == AU_W_TMAV && lane == 0) {
    tma_prefetch_map(&map_cv);
    tma_prefetch_map(&map_sv);
  }
  if (warp == AU_W_QK) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // tensor memory columns: O of row tile w at 128 w; its scores at 256 + 128 w, over whose first 64 columns the weights go
  if (!early) pdl_wait();        // (see k_attn_umma)

  const int r0 = __ldcg(sd.row_off + b);
  const int Qn = __ldcg(sd.row_off + b + 1) - r0;
  const int pos_tile = AU_BM / G;                       // whole query positions of G heads each per row tile
  const int pos0 = (int)blockIdx.x * 2 * pos_tile;
  const int n_w = pos0 >= Qn ? 0 : pos0 + pos_tile >= Qn ? 1 : 2;        // row tiles with rows
  const int F = __ldcg(sd.F + b) + (inplace ? Qn : 0);
  const int n_c = (F + AU_BN - 1) / AU_BN, n_s = inplace ? 0 : (Qn + AU_BN - 1) / AU_BN;
  const int n_tiles = n_w > 0 ? n_c + n_s : 0;
  const int ldq = n_heads * DH;

  if (warp == AU_W_TMA || warp == AU_W_TMAV) {
    // ---------------- TMA producers: one warp streams the K tiles, another the V tiles ----------------
    const bool is_v = warp == AU_W_TMAV;
    const int full = is_v ? B_VF : B_KF, empty = is_v ? B_VE : B_KE;
    auto load_tile = [&](int t) {
      if (elect_one()) {
        const int s = t & 1;
        mbar_expect_tx(bar(full + s), AU_TILE);
        const uint32_t dst = smem_u32(KVs + (size_t)s * 2 * AU_TILE) + (is_v ? AU_TILE : 0);
        const bool cache = t < n_c;
        const int row = cache ? b * max_len + t * AU_BN : r0 + (t - n_c) * AU_BN;
        const CUtensorMap* mp = cache ? (is_v ? &map_cv : &map_ck) : (is_v ? &map_sv : &map_sk);
        tma_load_2d(dst, mp, kvh * DH, row, bar(full + s));
        tma_load_2d(dst + AU_ATOM, mp, kvh * DH + 64, row, bar(full + s));
      }
      __syncwarp();
    };
    int issued = 0;
    if (early)
      while (issued < min(2, n_tiles) && (inplace ? (issued + 1) * AU_BN <= F - Qn : issued < n_c)) load_tile(issued++);
    pdl_wait();
    if (!is_v && n_tiles > 0 && elect_one()) {
      mbar_expect_tx(bar(B_Q), (uint32_t)(n_w * pos_tile * G * 256));
      for (int w = 0; w < n_w; ++w) {
        tma_load_5d_q(smem_u32(Qs) + w * AU_TILE, &map_q, kvh, r0 + pos0 + w * pos_tile, 0, bar(B_Q));
        tma_load_5d_q(smem_u32(Qs) + w * AU_TILE + AU_ATOM, &map_q, kvh, r0 + pos0 + w * pos_tile, 1, bar(B_Q));
      }
    }
    __syncwarp();
    for (int t = issued; t < n_tiles; ++t) {
      if (!__all_sync(0xffffffffu, mbar_wait(bar(empty + (t & 1)), ((uint32_t)(t >> 1) & 1u) ^ 1u, abort_flag))) {
        if (lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(status, 1u); status[1] = 31u; }
        break;
      }
      load_tile(t);
      ++issued;
    }
    // do not leave while copies may still be landing in this CTA's shared memory
    volatile uint32_t no_abort = 0;
    if (!is_v && n_tiles > 0) mbar_wait(bar(B_Q), 0u, &no_abort);
    for (int t = issued > 2 ? issued - 2 : 0; t < issued; ++t) mbar_wait(bar(full + (t & 1)), (uint32_t)(t >> 1) & 1u, &no_abort);
  } else if (warp == AU_W_QK) {
    // ---------------- MMA issuer (the whole warp waits, one elected thread issues) ----------------
    pdl_wait();
    constexpr uint32_t idesc_qk = make_idesc(AU_BN), idesc_pv = make_idesc(DH) | (1u << 16);      // P V: B (V) is MN-major
    bool ok = true;
    auto await = [&](bool got, unsigned site) {
      ok = __all_sync(0xffffffffu, got);
      if (!ok && lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(status, 1u); status[1] = site; }
      tc_fence_after();
      return ok;
    };
    auto qk = [&](int t, int w) {              // S_w = Q_w K^T of tile t
      if (elect_one()) {
        const uint32_t kd = smem_u32(KVs + (size_t)(t & 1) * 2 * AU_TILE), qd = smem_u32(Qs) + w * AU_TILE;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          tc_mma_f16(tmem_base + 256u + 128u * w, make_smem_desc(qd + (k >> 2) * AU_ATOM) + (uint64_t)(2 * (k & 3)),
                     make_smem_desc(kd + (k >> 2) * AU_ATOM) + (uint64_t)(2 * (k & 3)), idesc_qk, k ? 1u : 0u);
        tc_commit(bar(B_SF + w));
        if (w == n_w - 1) tc_commit(bar(B_KE + (t & 1)));
      }
      __syncwarp();
    };
    if (n_tiles > 0 && await(mbar_wait(bar(B_Q), 0u, abort_flag) && mbar_wait(bar(B_KF), 0u, abort_flag), 32u))
      for (int w = 0; w < n_w; ++w) qk(0, w);
    for (int t = 0; t < n_tiles && ok; ++t) {
      const uint32_t sp = (uint32_t)(t >> 1) & 1u;            // parity of the tile's stage
      if (!await(mbar_wait(bar(B_VF + (t & 1)), sp, abort_flag), 33u)) break;
      for (int w = 0; w < n_w; ++w) {
        if (!await(mbar_wait(bar(B_PR + w), (uint32_t)t & 1u, abort_flag), 34u)) break;
        if (elect_one()) {
          const uint32_t vd = smem_u32(KVs + (size_t)(t & 1) * 2 * AU_TILE) + AU_TILE;
#pragma unroll
          for (int k = 0; k < 8; ++k)              // 16 keys per step: 8 columns of packed weights
            tc_mma_f16_ts(tmem_base + 128u * w, tmem_base + 256u + 128u * w + 8u * k, make_smem_desc_mn(vd) + (uint64_t)(k * (2048 >> 4)), idesc_pv,
                          (t | k) ? 1u : 0u);
          if (w == n_w - 1) tc_commit(bar(B_VE + (t & 1)));
          if (t == n_tiles - 1) tc_commit(bar(B_PD + w));
        }
        __syncwarp();
        if (t + 1 < n_tiles) {
          if (w == 0 && !await(mbar_wait(bar(B_KF + ((t + 1) & 1)), (uint32_t)((t + 1) >> 1) & 1u, abort_flag), 35u)) break;
          qk(t + 1, w);
        }
      }
    }
  } else if (warp < 8) {
    // ---------------- softmax, one row per thread; group w = row tile w ----------------
    pdl_wait();
    const int w = warp >> 2, r = threadIdx.x & 127;
    const uint32_t lane_base = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t s_col = lane_base + 256u + 128u * w, o_col = lane_base + 128u * w;
    const int tiles = w < n_w ? n_tiles : 0;
    float m_used = -INFINITY, l = 0.f;
    bool ok = true;
    for (int t = 0; t < tiles; ++t) {
      if (!__all_sync(0xffffffffu, mbar_wait(bar(B_SF + w), (uint32_t)t & 1u, abort_flag))) {
        if (lane == 0 && !*abort_flag) { *abort_flag = 1; atomicExch(status, 1u); status[1] = 36u; }
        ok = false;
        break;
      }
      tc_fence_after();
      const int valid_keys = t < n_c ? min(AU_BN, F - t * AU_BN) : min(AU_BN, Qn - (t - n_c) * AU_BN);
      __syncwarp();                                     // the loads below are collective
      float sv[AU_BN];
#pragma unroll
      for (int c = 0; c < AU_BN; c += 16) tc_ld16_nowait(s_col + (uint32_t)c, sv + c);
      tc_wait_ld();
#pragma unroll
      for (int c = 0; c < AU_BN; c += 16) tc_pin16p(sv + c);
      if (valid_keys < AU_BN) {
#pragma unroll
        for (int i = 0; i < AU_BN; ++i)
          if (i >= valid_keys) sv[i] = -INFINITY;
      }
      float m4[4] = {sv[0], sv[1], sv[2], sv[3]};
#pragma unroll
      for (int i = 4; i < AU_BN; i += 8) {
#pragma unroll
        for (int k = 0; k < 4; ++k) m4[k] = fmaxf(fmaxf(m4[k], sv[i + k]), i + 4 + k < AU_BN ? sv[i + 4 + k] : sv[i + k]);
      }
      const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * scale_log2;
      float corr = 1.f;
      bool raise = false;
      if (mx > m_used + (t < 4 ? 0.25f : 8.f)) {        // also the first tile (m_used = -inf)
        corr = ex2_approx(m_used - mx);
        m_used = mx;
        raise = t > 0;
      }
      if (__any_sync(0xffffffffu, raise)) {             // rare after the first tiles: rescale the accumulator rows (the previous
#pragma unroll 1                                        // P V came before the scores in the tensor pipe)
        for (int c = 0; c < DH; c += 16) {
          float v[16];
          tc_ld16(o_col + (uint32_t)c, v);
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] *= corr;
          tc_st16(o_col + (uint32_t)c, v);
        }
      }
      // The tile's V rows past the last key hold whatever lies behind it, and 0 x NaN = NaN would reach every output row: both groups
      // clear them ahead of their own P V.
      if (valid_keys < AU_BN && r >= valid_keys && mbar_wait(bar(B_VF + (t & 1)), (uint32_t)(t >> 1) & 1u, abort_flag)) {
        uint8_t* vrow = KVs + (size_t)(t & 1) * 2 * AU_TILE + AU_TILE + (r >> 3) * 1024 + (r & 7) * 128;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          *reinterpret_cast<uint4*>(vrow + 16 * c) = make_uint4(0u, 0u, 0u, 0u);
          *reinterpret_cast<uint4*>(vrow + AU_ATOM + 16 * c) = make_uint4(0u, 0u, 0u, 0u);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      __syncwarp();
      // exponentials, packed in pairs over the scores' columns
      const float neg_m = -m_used;
      const f32x2 sc2 = f2_pack(scale_log2, scale_log2), nm2 = f2_pack(neg_m, neg_m);
      f32x2 sum2[2] = {0ull, 0ull};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t pk[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const f32x2 x2 = f2_fma(f2_pack(sv[32 * c + 2 * j], sv[32 * c + 2 * j + 1]), sc2, nm2);
          float p0, p1;
          f2_unpack(x2, p0, p1);
          p0 = ex2_approx(p0);
          p1 = ex2_approx(p1);
          const __nv_bfloat162 pb = __floats2bfloat162_rn(p0, p1);
          pk[j] = *reinterpret_cast<const uint32_t*>(&pb);
          sum2[j & 1] = f2_add(sum2[j & 1], f2_pack(__uint_as_float(pk[j] << 16), __uint_as_float(pk[j] & 0xffff0000u)));
        }
        tc_st16u(s_col + (uint32_t)(16 * c), pk);
      }
      float sa, sb;
      f2_unpack(f2_add(sum2[0], sum2[1]), sa, sb);
      l = l * corr + (sa + sb);
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(B_PR + w));        // P_w ready
    }
    const bool have = __all_sync(0xffffffffu, ok && tiles > 0 && mbar_wait(bar(B_PD + w), 0u, abort_flag));
    if (have) {
      tc_fence_after();
      const float inv = __fdividef(1.f, l);
      const int qi = pos0 + w * pos_tile + r / G, hg = r % G;
      const bool valid = r < pos_tile * G && qi < Qn;
      uint4* dst = reinterpret_cast<uint4*>(out + (size_t)(r0 + qi) * ldq + (kvh * G + hg) * DH);
#pragma unroll 1
      for (int c = 0; c < DH; c += 32) {
        float v[16], u[16];
        __syncwarp();
        tc_ld16_nowait(o_col + (uint32_t)c, v);
        tc_ld16_nowait(o_col + (uint32_t)(c + 16), u);
        tc_wait_ld();
        tc_pin16(v);
        tc_pin16(u);
        if (valid) {
#pragma unroll
          for (int i = 0; i < 16; ++i) { v[i] *= inv; u[i] *= inv; }
          dst[c >> 3] = pack8(v);
          dst[(c >> 3) + 1] = pack8(v + 8);
          dst[(c >> 3) + 2] = pack8(u);
          dst[(c >> 3) + 3] = pack8(u + 8);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == AU_W_QK) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

}  // namespace lsp
