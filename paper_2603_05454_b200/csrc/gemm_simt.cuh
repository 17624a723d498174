// CUDA-core GEMM (fp32 accumulate) with the shared epilogues.  It is the compute path of fp32 models and the reference
// implementation the tcgen05 kernels can be switched against.
//
// k_gemm_simt: 64 x 64 output tiles, one CTA each, for problems that fill the SMs with them.
// k_gemm_simt_split: the fp32 models it serves are small, so a launch is mostly bound by latency, not arithmetic: few output
// tiles, each with a serial loop over K.  Tiles are therefore small (32 x 32 outputs, or 16 x 64 for the reducing head
// epilogue) and the eight warps of a CTA split K: warp w takes the 16-element steps w, w + 8, ... of the whole tile, loading the next step's operands while it
// multiplies this one's; the eight partial tiles are summed in warp order through shared memory (the same order every time)
// and each thread finishes four neighbouring outputs (two pairs).
// Measured (B200, fp32, us, k_gemm_simt -> k_gemm_simt_split): 65 x 384 (K 256) 15.2 -> 5.9, 128 x 256 (K 1024) 51 -> 14.8,
// 300 x 2048 (K 1024; 160 tiles of 64 x 64) 97 -> 53, 1024 x 4096 (K 4096; 1024 tiles) 1007 -> over 1100: the line is drawn at
// two 64 x 64 tiles per SM.  Four neighbouring lanes load a row's 64 bytes of a step (a row per lane cost four times the
// cache lines per instruction: 18 us instead of 14.8), and sixteen warps per CTA gained nothing.  Near the line two launches lose: the
// head at 250 rows of 2048 ids (K 256) 22.0 -> 25.9 and bf16 1032 x 2 x 1024 (K 256) 49 -> 52; the split sums are the more exact ones
// (p_max of that head 1.2e-6 from 64 bits, 4.4e-6 before), so the line stays.
#pragma once
#include "cluster.cuh"
#include "epilogues.cuh"

namespace lsp {

__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const bf16* p) {
  const uint2 t = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&t.x);
  const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&t.y);
  return make_float4(__low2float(a), __high2float(a), __low2float(b), __high2float(b));
}

constexpr int SG_KS = 16;         // K elements per step
constexpr int SG_WARPS = 8;
constexpr int SG_MAX_SLICES = 4;
// K slices of a tile (the CTAs of a cluster): where the tiles leave SMs idle, as long as every warp keeps two steps (a slice of one
// step per warp would cost the sum across the cluster, over a microsecond, for less than it saves).
inline int simt_slices(long tiles, int K, int n_sm, bool reduce) {
  int s = 1;
  while (!reduce && 2 * s <= SG_MAX_SLICES && 2 * s * tiles <= n_sm && K / SG_KS >= 2 * s * SG_WARPS * 2) s *= 2;
  return s;
}
// tile: rows x weight rows (a paired epilogue's tile holds half as many pairs); the head reduces 64 columns per partial
template <typename Epi> struct SimtTile {
  static constexpr int BM = Epi::kReduce ? 16 : 32, BN = Epi::kReduce ? 64 : 32;
  static constexpr int PER_TILE = Epi::kDual ? BN / 2 : BN;
};
constexpr int SG_HEAD_BN = 64;    // columns per partial of the head, in both kernels

// grid = (ceil(NP / PER_TILE) * slices, ceil(M / BM)), block = 256, clusters of slices CTAs along x: the K slices of a tile.  A: [M, K];
// W0/W1: [*, K] row-major.  kSliced: slices > 1 (a kernel of its own: with the slices' arithmetic and sums as run-time branches a launch
// without them took 0.2 to 0.3 us more: fp32, K 256, 33 x 1024 7.2 -> 7.5, 64 x 2 x 1024 8.3 -> 8.6).
template <typename T, typename Epi, bool kSliced>
__global__ void __launch_bounds__(32 * SG_WARPS) k_gemm_simt_split(const T* A, const T* __restrict__ W0,
                                                                   const T* __restrict__ W1, int M, int NP, int K, int slices, Epi epi) {
  constexpr int BM = SimtTile<Epi>::BM, BN = SimtTile<Epi>::BN, PT = SimtTile<Epi>::PER_TILE;
  constexpr int LA = BM + 4, LB = BN + 4;                       // padded leading dimensions
  constexpr int NA = BM * SG_KS / 4 / 32, NB = BN * SG_KS / 4 / 32;      // 4-element vectors per lane and step
  constexpr int WARP_F = SG_KS * (LA + LB);                     // floats of a warp's stage
  constexpr int RED_F = BM * BN;                                // floats of a partial tile
  __shared__ __align__(16) float sm[SG_WARPS * (WARP_F > RED_F ? WARP_F : RED_F)];
  pdl_begin();
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const int tile = kSliced ? blockIdx.x / (unsigned)slices : blockIdx.x, slice = kSliced ? blockIdx.x % (unsigned)slices : 0;
  const int m0 = blockIdx.y * BM, j0 = tile * PT;
  float* As = sm + w * WARP_F;
  float* Bs = As + SG_KS * LA;
  // operand rows of this lane's vectors, four neighbouring lanes to a row's 16 elements (null past the edges)
  static_assert(SG_KS == 16, "four vectors per row");
  const T* ap[NA];
  const T* bp[NB];
#pragma unroll
  for (int i = 0; i < NA; ++i) {
    const int v = lane + 32 * i, m = m0 + (v >> 2);
    ap[i] = m < M ? A + (size_t)m * K + (v & 3) * 4 : nullptr;
  }
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int v = lane + 32 * i, c = v >> 2;
    const int j = j0 + (Epi::kDual ? c % PT : c);
    const T* row = (Epi::kDual && c >= PT) ? W1 + (size_t)epi.row1(j) * K : W0 + (size_t)epi.row0(j) * K;
    bp[i] = j < NP ? row + (v & 3) * 4 : nullptr;
  }
  const int rg = lane / (BN / 8), cg = lane % (BN / 8);         // rows 4 rg .., columns 4 cg .. and BN / 2 + 4 cg ..
  float acc[4][8] = {};
  float4 av[NA], bv[NB];
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  auto load = [&](int k0) {
#pragma unroll
    for (int i = 0; i < NA; ++i) av[i] = ap[i] ? load4(ap[i] + k0) : zero;
#pragma unroll
    for (int i = 0; i < NB; ++i) bv[i] = bp[i] ? load4(bp[i] + k0) : zero;
  };
  const int lo = kSliced ? K / SG_KS * slice / slices : 0, steps = kSliced ? K / SG_KS * (slice + 1) / slices : K / SG_KS;
  if (lo + w < steps) load((lo + w) * SG_KS);
  for (int s = lo + w; s < steps; s += SG_WARPS) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int v = lane + 32 * i;
      float* d = As + (v & 3) * 4 * LA + (v >> 2);
      d[0] = av[i].x; d[LA] = av[i].y; d[2 * LA] = av[i].z; d[3 * LA] = av[i].w;
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int v = lane + 32 * i;
      float* d = Bs + (v & 3) * 4 * LB + (v >> 2);
      d[0] = bv[i].x; d[LB] = bv[i].y; d[2 * LB] = bv[i].z; d[3 * LB] = bv[i].w;
    }
    __syncwarp();
    if (s + SG_WARPS < steps) load((s + SG_WARPS) * SG_KS);
#pragma unroll
    for (int k = 0; k < SG_KS; ++k) {
      const float4 a = *reinterpret_cast<const float4*>(As + k * LA + 4 * rg);
      const float4 b0 = *reinterpret_cast<const float4*>(Bs + k * LB + 4 * cg);
      const float4 b1 = *reinterpret_cast<const float4*>(Bs + k * LB + BN / 2 + 4 * cg);
      const float ar[4] = {a.x, a.y, a.z, a.w}, br[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(ar[i], br[j], acc[i][j]);
    }
  }
  __syncthreads();                       // the stages become the partial tiles
  float* red = sm + w * RED_F;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    *reinterpret_cast<float4*>(red + (4 * rg + i) * BN + 4 * cg) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    *reinterpret_cast<float4*>(red + (4 * rg + i) * BN + BN / 2 + 4 * cg) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
  }
  __syncthreads();
  constexpr int TPR = BN / 4;            // threads per output row
  const int row = t / TPR, m = m0 + row;
  // K slices: every CTA leaves its sums in its shared memory, and the first one adds them in slice (= K) order (true: this CTA
  // finishes the tile)
  auto sum_slices = [&](float (&v)[4]) -> bool {
    if constexpr (!kSliced) return true;
    float4* out = reinterpret_cast<float4*>(sm);
    __syncthreads();                     // the warps' partial tiles have been read
    if (slice > 0) out[t] = make_float4(v[0], v[1], v[2], v[3]);
    cluster_sync();
    if (slice == 0) {
      const uint32_t a = smem_u32(out + t);
      float4 p[SG_MAX_SLICES - 1];
#pragma unroll
      for (int x = 1; x < SG_MAX_SLICES; ++x)
        if (x < slices) p[x - 1] = ld_cluster_f4(cluster_map(a, (unsigned)x));
#pragma unroll
      for (int x = 1; x < SG_MAX_SLICES; ++x)
        if (x < slices) { v[0] += p[x - 1].x; v[1] += p[x - 1].y; v[2] += p[x - 1].z; v[3] += p[x - 1].w; }
    }
    cluster_sync();                      // nobody leaves while its sums may still be read
    return slice == 0;
  };
  if constexpr (Epi::kDual) {
    const int p = (t % TPR) * 2;         // two pairs: columns p, p + 1 and PT + p, PT + p + 1
    float a0[2] = {}, a1[2] = {};
#pragma unroll
    for (int x = 0; x < SG_WARPS; ++x) {
      const float* r = sm + x * RED_F + row * BN + p;
      const float2 u = *reinterpret_cast<const float2*>(r), v = *reinterpret_cast<const float2*>(r + PT);
      a0[0] += u.x; a0[1] += u.y; a1[0] += v.x; a1[1] += v.y;
    }
    float a[4] = {a0[0], a0[1], a1[0], a1[1]};
    const bool mine = sum_slices(a);
    a0[0] = a[0]; a0[1] = a[1]; a1[0] = a[2]; a1[1] = a[3];
    if (mine && m < M) {
#pragma unroll
      for (int e = 0; e < 2; ++e)
        if (j0 + p + e < NP) epi.elem(m, j0 + p + e, a0[e], a1[e]);
    }
  } else {
    const int c = (t % TPR) * 4;
    float a[4] = {};
#pragma unroll
    for (int x = 0; x < SG_WARPS; ++x) {
      const float4 u = *reinterpret_cast<const float4*>(sm + x * RED_F + row * BN + c);
      a[0] += u.x; a[1] += u.y; a[2] += u.z; a[3] += u.w;
    }
    const bool mine = sum_slices(a);
    if constexpr (Epi::kReduce) {
      Top2 r = top2_empty();
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (epi.valid(j0 + c + e)) top2_push(r, a[e], j0 + c + e);
#pragma unroll
      for (int o = 1; o < TPR; o <<= 1) r = top2_merge(r, top2_shfl_xor(r, o));
      if (t % TPR == 0 && m < M) epi.part[(size_t)m * epi.n_tiles + tile] = r;
    } else if (mine && m < M) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j0 + c + e < NP) epi.elem(m, j0 + c + e, a[e], 0.f);
    }
  }
}

__device__ __forceinline__ void load4(const float* p, float (&v)[4]) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void load4(const bf16* p, float (&v)[4]) {
  const uint2 t = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&t.x);
  const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&t.y);
  v[0] = __low2float(a); v[1] = __high2float(a); v[2] = __low2float(b); v[3] = __high2float(b);
}

constexpr int SG_BM = 64, SG_BN = SG_HEAD_BN, SG_BK = 16;

// grid = (ceil(NP / 64), ceil(M / 64)), block = 256.  A: [M, K]; W0/W1: [*, K] row-major.
template <typename T, typename Epi>
__global__ void __launch_bounds__(256) k_gemm_simt(const T* A, const T* __restrict__ W0,
                                                   const T* __restrict__ W1, int M, int NP, int K, Epi epi) {
  __shared__ float As[SG_BK][SG_BM + 4];
  __shared__ float B0s[SG_BK][SG_BN + 4];
  __shared__ float B1s[Epi::kDual ? SG_BK : 1][SG_BN + 4];
  pdl_begin();
  const int t = threadIdx.x;
  const int m0 = blockIdx.y * SG_BM, j0 = blockIdx.x * SG_BN;
  const int lrow = t >> 2, lk = (t & 3) * 4;
  const int am = m0 + lrow;
  const int bj = j0 + lrow;
  const T* ap = (am < M) ? A + (size_t)am * K + lk : nullptr;
  const T* b0p = (bj < NP) ? W0 + (size_t)epi.row0(bj) * K + lk : nullptr;
  const T* b1p = (Epi::kDual && bj < NP) ? W1 + (size_t)epi.row1(bj) * K + lk : nullptr;
  const int ty = t >> 4, tx = t & 15;
  float acc0[4][4] = {}, acc1[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += SG_BK) {
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (ap) load4(ap + k0, v);
#pragma unroll
    for (int i = 0; i < 4; ++i) As[lk + i][lrow] = v[i];
    float w[4] = {0.f, 0.f, 0.f, 0.f};
    if (b0p) load4(b0p + k0, w);
#pragma unroll
    for (int i = 0; i < 4; ++i) B0s[lk + i][lrow] = w[i];
    if (Epi::kDual) {
      float u[4] = {0.f, 0.f, 0.f, 0.f};
      if (b1p) load4(b1p + k0, u);
#pragma unroll
      for (int i = 0; i < 4; ++i) B1s[lk + i][lrow] = u[i];
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < SG_BK; ++kk) {
      float a[4], b0[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) { a[i] = As[kk][ty * 4 + i]; b0[i] = B0s[kk][tx * 4 + i]; }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc0[i][j] = fmaf(a[i], b0[j], acc0[i][j]);
      if (Epi::kDual) {
        float b1[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) b1[i] = B1s[kk][tx * 4 + i];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc1[i][j] = fmaf(a[i], b1[j], acc1[i][j]);
      }
    }
    __syncthreads();
  }
  if constexpr (Epi::kReduce) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + ty * 4 + i;
      Top2 r = top2_empty();
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int col = j0 + tx * 4 + j;
        if (epi.valid(col)) top2_push(r, acc0[i][j], col);
      }
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) r = top2_merge(r, top2_shfl_xor(r, o));
      if (tx == 0 && m < M) epi.part[(size_t)m * epi.n_tiles + blockIdx.x] = r;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + ty * 4 + i;
      if (m >= M) continue;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int col = j0 + tx * 4 + j;
        if (col < NP) epi.elem(m, col, acc0[i][j], acc1[i][j]);
      }
    }
  }
}

}  // namespace lsp
