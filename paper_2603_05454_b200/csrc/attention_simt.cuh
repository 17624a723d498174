// CUDA-core flash-style attention: suffix queries over [contiguous prefix cache | this pass's staged rows].
// Non-causal: every query row sees every key (the bidirectional lookahead of Sec. 3.2).  fp32 arithmetic with
// an online softmax; used for fp32 models and as the switchable reference of the tensor-core kernel.
#pragma once
#include "common.cuh"

namespace lsp {

// Queries per block: 4 per warp where that still gives a block per SM, else 1 per warp (the K/V tile is then used by fewer
// queries, but a small pass is bound by one block's serial walk over the keys: tiny model, 26 -> 19 us a launch; with vector
// loads a tile ahead and four dot-product chains 12).  The loads a tile ahead pay for four queries too, whose registers they fill
// (166 at 64, 255 at 128): fp32, 4 x 258 rows over 958 keys, 32 heads of 128 4.53 -> 1.57 ms, 16 heads of 64 0.74 -> 0.38; bf16
// alike.
__device__ __forceinline__ float4 as_load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 as_load4(const bf16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&u.x), b = *reinterpret_cast<const __nv_bfloat162*>(&u.y);
  return make_float4(__low2float(a), __high2float(a), __low2float(b), __high2float(b));
}
constexpr int AS_BK = 32;   // keys per tile (one per lane)

// grid = (ceil(max_rows_per_seq / (4 QW)), n_heads, batch), block = 128; QW queries per warp.
// q: [M, n_heads*DH]; cache_k/v: this layer's planes [batch_max][max_len][n_kv*DH]; stage_k/v: this layer's
// staged planes [M][n_kv*DH]; out: [M, n_heads*DH].
template <typename T, int DH, int QW>
__global__ void __launch_bounds__(128) k_attn_simt(const T* q, const T* cache_k,
                                                   const T* cache_v, const T* stage_k,
                                                   const T* stage_v, T* __restrict__ out, StepDesc sd,
                                                   int n_heads, int n_kv_heads, size_t cache_seq_elems,
                                                   float scale, int inplace) {
  constexpr int AS_BQ = 4 * QW;
  __shared__ float Qs[AS_BQ][DH];
  __shared__ float Ks[AS_BK][DH + 1];
  __shared__ __align__(16) float Vs[AS_BK][DH];
  pdl_begin();
  const int b = blockIdx.z, h = blockIdx.y;
  const int r0 = sd.row_off[b];
  const int Qn = sd.row_off[b + 1] - r0;
  const int q0 = blockIdx.x * AS_BQ;
  if (q0 >= Qn) return;
  const int S = sd.F[b] + Qn;
  const int F = inplace ? S : sd.F[b];      // in-place layout: this pass's K/V rows already sit behind the prefix in the cache
  const int kvh = h / (n_heads / n_kv_heads);
  const int ldq = n_heads * DH, ldkv = n_kv_heads * DH;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  for (int i = t; i < AS_BQ * DH; i += 128) {
    const int qi = i / DH, d = i % DH;
    Qs[qi][d] = (q0 + qi < Qn) ? to_f(q[(size_t)(r0 + q0 + qi) * ldq + h * DH + d]) : 0.f;
  }
  constexpr int NC = DH / 32;
  float acc[QW][NC];
  float m_run[QW], l_run[QW];
#pragma unroll
  for (int i = 0; i < QW; ++i) {
    m_run[i] = -INFINITY;
    l_run[i] = 0.f;
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[i][c] = 0.f;
  }
  const T* ck = cache_k + (size_t)b * cache_seq_elems + kvh * DH;
  const T* cv = cache_v + (size_t)b * cache_seq_elems + kvh * DH;
  const T* sk = stage_k + (size_t)r0 * ldkv + kvh * DH;
  const T* sv = stage_v + (size_t)r0 * ldkv + kvh * DH;
  // A tile's keys and values: vector i of thread t is elements 4 (t % (DH / 4)) .. of key t / (DH / 4) + i * KPI.  The next tile's
  // are fetched while this one's are used.
  constexpr int VPR = DH / 4, KPI = 128 / VPR, NV = AS_BK / KPI;
  float4 kreg[NV], vreg[NV];
  const int vk = t / VPR, ve = (t % VPR) * 4;
  auto fetch = [&](int s0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int s = s0 + vk + i * KPI;
      const T* kp = nullptr;
      const T* vp = nullptr;
      if (s < F) { kp = ck + (size_t)s * ldkv; vp = cv + (size_t)s * ldkv; }
      else if (s < S) { kp = sk + (size_t)(s - F) * ldkv; vp = sv + (size_t)(s - F) * ldkv; }
      kreg[i] = kp ? as_load4(kp + ve) : make_float4(0.f, 0.f, 0.f, 0.f);
      vreg[i] = vp ? as_load4(vp + ve) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  fetch(0);
  for (int s0 = 0; s0 < S; s0 += AS_BK) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int key = vk + i * KPI;
      Ks[key][ve] = kreg[i].x; Ks[key][ve + 1] = kreg[i].y; Ks[key][ve + 2] = kreg[i].z; Ks[key][ve + 3] = kreg[i].w;
      *reinterpret_cast<float4*>(&Vs[key][ve]) = vreg[i];
    }
    __syncthreads();
    if (s0 + AS_BK < S) fetch(s0 + AS_BK);
    const bool kvalid = (s0 + lane) < S;
#pragma unroll
    for (int i = 0; i < QW; ++i) {
      const int qi = w * QW + i;
      float d4[4] = {0.f, 0.f, 0.f, 0.f};                     // (four chains: one would be DH dependent steps)
#pragma unroll 4
      for (int d = 0; d < DH; d += 4) {
#pragma unroll
        for (int e = 0; e < 4; ++e) d4[e] = fmaf(Qs[qi][d + e], Ks[lane][d + e], d4[e]);
      }
      const float dot = (d4[0] + d4[1]) + (d4[2] + d4[3]);
      const float sc = kvalid ? dot * scale : -INFINITY;
      const float m_new = fmaxf(m_run[i], warp_max(sc));
      const float p = kvalid ? __expf(sc - m_new) : 0.f;
      const float corr = __expf(m_run[i] - m_new);
      l_run[i] = l_run[i] * corr + warp_sum(p);
      m_run[i] = m_new;
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[i][c] *= corr;
      for (int k = 0; k < AS_BK; ++k) {
        const float pk = __shfl_sync(0xffffffffu, p, k);
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[i][c] = fmaf(pk, Vs[k][lane + 32 * c], acc[i][c]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < QW; ++i) {
    const int qq = q0 + w * QW + i;
    if (qq >= Qn) continue;
    const float inv = 1.f / l_run[i];
#pragma unroll
    for (int c = 0; c < NC; ++c)
      out[(size_t)(r0 + qq) * ldq + h * DH + lane + 32 * c] = from_f<T>(acc[i][c] * inv);
  }
}

// Small passes: one query per CTA, its keys split over the four warps in tiles of 32 (one key per lane).  A lane reads its key's row and
// the warp the tile's value rows straight from memory, all requested before the first is used, and the warps' partial results are merged
// at the end: with 128 keys every warp has one tile, where the kernel above walks four in series.  Every query reads all keys and
// values itself, so this is for as many CTAs as are resident at once (the dispatch: at most three per SM).
template <typename T, int DH>
__global__ void __launch_bounds__(128) k_attn_simt_split(const T* q, const T* cache_k, const T* cache_v, const T* stage_k, const T* stage_v,
                                                         T* __restrict__ out, StepDesc sd, int n_heads, int n_kv_heads,
                                                         size_t cache_seq_elems, float scale, int inplace) {
  constexpr int NV = DH / 4, NC = DH / 32;             // 4-element vectors of a row; elements of the output per lane
  __shared__ __align__(16) float qs[4][DH];            // a copy per warp: no barrier before the merge
  __shared__ float part[4][DH], pm[4], pl[4];
  pdl_begin();
  const int b = blockIdx.z, h = blockIdx.y, qi = blockIdx.x;
  const int r0 = sd.row_off[b], Qn = sd.row_off[b + 1] - r0;
  if (qi >= Qn) return;
  const int S = sd.F[b] + Qn;
  const int F = inplace ? S : sd.F[b];      // in-place layout: this pass's K/V rows already sit behind the prefix in the cache
  const int kvh = h / (n_heads / n_kv_heads), ldq = n_heads * DH, ldkv = n_kv_heads * DH;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const T* ck = cache_k + (size_t)b * cache_seq_elems + kvh * DH;
  const T* cv = cache_v + (size_t)b * cache_seq_elems + kvh * DH;
  const T* sk = stage_k + (size_t)r0 * ldkv + kvh * DH;
  const T* sv = stage_v + (size_t)r0 * ldkv + kvh * DH;
  float qr[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) qr[c] = to_f(q[(size_t)(r0 + qi) * ldq + h * DH + lane + 32 * c]);
  float m = -INFINITY, l = 0.f, acc[NC] = {};
  for (int s0 = 32 * w; s0 < S; s0 += 128) {
    const int key = s0 + lane;
    const T* kp = key < F ? ck + (size_t)key * ldkv : sk + (size_t)(key < S ? key - F : 0) * ldkv;
    if (key >= S) kp = sk;                  // (a row of this pass, there is one)
    float4 kr[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) kr[i] = as_load4(kp + 4 * i);
    float v[32][NC];
    auto load_v = [&]() {
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const int kk = s0 + k;
        const T* vp = kk < F ? cv + (size_t)kk * ldkv : sv + (size_t)(kk - F) * ldkv;
#pragma unroll
        for (int c = 0; c < NC; ++c) v[k][c] = kk < S ? to_f(vp[lane + 32 * c]) : 0.f;
      }
    };
    if (DH == 64) load_v();                 // (with 128 elements a row the key's registers are needed first)
    if (s0 == 32 * w) {
#pragma unroll
      for (int c = 0; c < NC; ++c) qs[w][lane + 32 * c] = qr[c];
      __syncwarp();
    }
    float d4[4] = {};
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const float4 qv = *reinterpret_cast<const float4*>(qs[w] + 4 * i);
      d4[0] = fmaf(qv.x, kr[i].x, d4[0]);
      d4[1] = fmaf(qv.y, kr[i].y, d4[1]);
      d4[2] = fmaf(qv.z, kr[i].z, d4[2]);
      d4[3] = fmaf(qv.w, kr[i].w, d4[3]);
    }
    const float sc = key < S ? ((d4[0] + d4[1]) + (d4[2] + d4[3])) * scale : -INFINITY;
    // (a score that overflowed to -inf has no weight, also where a warp has met no other yet: the kernel above has by then unless it
    // is the first tile's)
    const float m_new = fmaxf(m, warp_max(sc));
    const float m_ref = m_new == -INFINITY ? 0.f : m_new;
    const float p = key < S ? __expf(sc - m_ref) : 0.f;
    const float corr = __expf(m - m_ref);
    l = l * corr + warp_sum(p);
    m = m_new;
    if (DH != 64) load_v();
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] *= corr;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const float pk = __shfl_sync(0xffffffffu, p, k);
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = fmaf(pk, v[k][c], acc[c]);
    }
  }
  if (lane == 0) { pm[w] = m; pl[w] = l; }
#pragma unroll
  for (int c = 0; c < NC; ++c) part[w][lane + 32 * c] = acc[c];
  __syncthreads();
  if (t < DH) {
    const float mx = fmaxf(fmaxf(pm[0], pm[1]), fmaxf(pm[2], pm[3]));
    float sum = 0.f, ls = 0.f;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const float f = pm[x] == -INFINITY ? 0.f : __expf(pm[x] - mx);
      ls += f * pl[x];
      sum += f * part[x][t];
    }
    out[(size_t)(r0 + qi) * ldq + h * DH + t] = from_f<T>(sum / ls);
  }
}

}  // namespace lsp
