// bf16 GEMM on the 5th-generation tensor cores (tcgen05) for sm_100a: the parts shared by every kernel that uses them.
//
//   acc[m, c] = sum_k A[m, k] * Wt[c, k]        A: [M, K] bf16 row-major, Wt: weight rows, K-major, fp32 accumulate
//
// This header holds the PTX wrappers (mbarrier with bounded waits, TMA tile loads (every CTA fetches its own tiles), tcgen05.mma /
// .commit / .ld), the shared-memory and instruction descriptors, the vectorised fused epilogues (store / residual /
// SwiGLU / rotary + K/V staging), the host state (tensor-map caches, tuning fields) and the dispatch that picks
// kernel and tile width.  The kernels are k_gemm_stream (gemm_stream.cuh, up to 128 rows) and k_gemm_pair (gemm_pair.cuh, more);
// the attention kernel (attention_umma.cuh) uses the same wrappers.
//
// The B tile is two blocks of BN/2 weight rows each (possibly from two tensors), so accumulator columns
// c and c + BN/2 of one thread hold the pair an element-wise fusion needs (gate/up, rotate-half partners).
// Every wait is bounded by wall-clock time; on expiry a kernel records (code, site) in a status word, lets
// all roles drain and returns, so a protocol error can never hang the device.
#pragma once
#include <cuda.h>

#include <map>
#include <set>
#include <string>
#include <tuple>

#include "epilogues.cuh"

namespace lsp {

constexpr int UM_BM = 128;
constexpr int UM_BK = 64;                 // bf16 elements = one 128-byte swizzle row
constexpr int UM_MAX_STAGES = 12;
constexpr uint64_t UM_WAIT_NS = 2000000000ull;   // 2 s

// ---- PTX wrappers -----------------------------------------------------------------------------------------
__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok;
}
// The same without suspending the thread.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false after limit_ns (default UM_WAIT_NS) or when another role has raised the abort flag.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                          uint64_t limit_ns = UM_WAIT_NS) {
  uint64_t t0 = 0;
  for (uint32_t spin = 0;; ++spin) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((spin & 1023u) == 1023u) {
      if (*abort_flag) return false;
      const uint64_t now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) return false;
    }
  }
}

// After a failure a stage may hold copies of one producer and none of the other, and its barrier then never completes.  Each producer
// stays this long (1 ms; a copy takes microseconds) behind its last copy instead, so that none lands in the memory of a CTA that is gone.
__device__ __forceinline__ void um_let_land() {
  const uint64_t t0 = globaltimer_ns();
  while (globaltimer_ns() - t0 < 1000000ull) {}
}

// Self-test of the bounded-wait protocol: one thread waits on a barrier that nobody ever arrives at, gives up after
// limit_ns and reports it exactly as the kernels' roles do: (code 1, site 99) in the status word.  Nothing else runs,
// nothing is in flight, the context stays usable.
__global__ void k_wait_selftest(unsigned* status, unsigned long long limit_ns) {
  __shared__ uint64_t never;
  __shared__ uint32_t no_abort;
  if (threadIdx.x == 0) {
    no_abort = 0;
    mbar_init(smem_u32(&never), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!mbar_wait(smem_u32(&never), 0u, &no_abort, (uint64_t)limit_ns)) {
      atomicExch(status, 1u);
      status[1] = 99u;
    }
  }
}
// Fetches a tensor map ahead of the first copy that uses it (about a microsecond of its latency).
__device__ __forceinline__ void tma_prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
// One box of a 5-D map (umma_map5): rows r0.. of blocks blk.., both halves, 64-element K atoms a0..
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, int r0, int blk, int half, int a0, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
      ::"r"(dst), "l"(map), "r"(0), "r"(r0), "r"(blk), "r"(half), "r"(a0), "r"(bar)
      : "memory");
}
// True in one thread of a converged warp.  A tcgen05.mma behind a lane test (if (lane == 0)) costs its issuer about 130 cycles
// whatever its width when a commit follows every fourth, behind elect.sync 88; a turn of a stage ring costs a producer or
// issuer about 300 ns in all, so stages are large and each operand of a stage is one copy.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(p));
  return p != 0;
}
// One box of a 4-D map (umma_map4): rows r0.. of block blk.., 64-element K atoms a0..
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int r0, int blk, int a0, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(map), "r"(0), "r"(r0), "r"(blk), "r"(a0), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                           uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 16 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// 16 consecutive fp32 columns of this thread's TMEM lane, without waiting: several loads can be in flight before one
// tc_wait_ld(); the destination must not be read before that wait.
__device__ __forceinline__ void tc_ld16_nowait(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// Placed after tc_wait_ld(): makes every later use of v depend on a statement that follows the wait, so that the compiler
// cannot schedule arithmetic on the loaded values ahead of it.
__device__ __forceinline__ void tc_pin16(float (&v)[16]) {
  asm volatile("" : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]), "+f"(v[8]),
               "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]));
}

// Shared-memory matrix descriptor for a K-major bf16 tile stored as rows of 128 bytes with the 128-byte swizzle:
// 8-row groups are 1024 bytes apart (stride byte offset); the leading byte offset is unused for this layout.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);        // start address, 16-byte units
  d |= (uint64_t)1 << 16;                          // leading byte offset (ignored with swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset
  d |= (uint64_t)1 << 46;                          // descriptor version for this architecture
  d |= (uint64_t)2 << 61;                          // layout: 128-byte swizzle
  return d;
}
// Instruction descriptor: D = f32, A = B = bf16, both K-major, M = 128, N = BN.
__host__ __device__ constexpr uint32_t make_idesc(int bn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(UM_BM >> 4) << 24);
}

// ---- vector helpers for the epilogues ------------------------------------------------------------------
__device__ __forceinline__ uint4 pack8(const float* v) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]);
  __nv_bfloat162 b = __floats2bfloat162_rn(v[2], v[3]);
  __nv_bfloat162 c = __floats2bfloat162_rn(v[4], v[5]);
  __nv_bfloat162 d = __floats2bfloat162_rn(v[6], v[7]);
  uint4 r;
  r.x = *reinterpret_cast<uint32_t*>(&a);
  r.y = *reinterpret_cast<uint32_t*>(&b);
  r.z = *reinterpret_cast<uint32_t*>(&c);
  r.w = *reinterpret_cast<uint32_t*>(&d);
  return r;
}
__device__ __forceinline__ void unpack8(const uint4& u, float* v) {
  const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = __low2float(p[i]);
    v[2 * i + 1] = __high2float(p[i]);
  }
}

// 16 consecutive pair indices j..j+15 of row m (a1 unused for plain epilogues).
__device__ __forceinline__ void epi16(const EpiStore<bf16>& e, int m, int j, const float* a0, const float*) {
  uint4* p = reinterpret_cast<uint4*>(e.out + (size_t)m * e.ld + j);
  p[0] = pack8(a0);
  p[1] = pack8(a0 + 8);
}
// What an epilogue reads from memory for 16 columns (or pairs), fetched ahead of the accumulators: EpiPre::load early, then
// epi16 with it.  Left to the epilogue itself, one L2 round trip (two for the rotary table, which is indexed by a loaded row
// position) per chunk of 16 columns lies behind the last MMA: 5 us of a QKV projection, 2 to 3 of an O or down projection.
template <typename Epi>
struct EpiPre {
  __device__ __forceinline__ void load(const Epi&, int, int) {}
};
template <>
struct EpiPre<EpiResidual<bf16>> {
  uint4 x[2];
  __device__ __forceinline__ void load(const EpiResidual<bf16>& e, int m, int j) {
    const uint4* p = reinterpret_cast<const uint4*>(e.x + (size_t)m * e.ld + j);
    x[0] = p[0];
    x[1] = p[1];
  }
};
template <>
struct EpiPre<EpiQKVRope<bf16>> {
  float4 c[8];        // (cos, sin) of 16 frequencies
  __device__ __forceinline__ void load(const EpiQKVRope<bf16>& e, int m, int j) {
    const int h = j / e.half, i = j % e.half;
    if (h < e.n_heads + e.n_kv_heads) {
      const float4* c4 = reinterpret_cast<const float4*>(e.cs + (size_t)e.row_pos[m] * e.half + i);
#pragma unroll
      for (int q = 0; q < 8; ++q) c[q] = __ldg(c4 + q);
    }
  }
};
template <typename Epi>
__device__ __forceinline__ void epi16(const Epi& e, int m, int j, const float* a0, const float* a1, const EpiPre<Epi>&) {
  epi16(e, m, j, a0, a1);
}
__device__ __forceinline__ void epi16(const EpiResidual<bf16>& e, int m, int j, const float* a0, const float*,
                                      const EpiPre<EpiResidual<bf16>>& pre) {
  uint4* p = reinterpret_cast<uint4*>(e.x + (size_t)m * e.ld + j);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float x[8];
    unpack8(pre.x[h], x);
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] += a0[8 * h + i];
    p[h] = pack8(x);
  }
}
__device__ __forceinline__ void epi16(const EpiResidual<bf16>& e, int m, int j, const float* a0, const float* a1) {
  EpiPre<EpiResidual<bf16>> pre;
  pre.load(e, m, j);
  epi16(e, m, j, a0, a1, pre);
}
__device__ __forceinline__ void epi16(const EpiSwiGLU<bf16>& e, int m, int j, const float* g, const float* u) {
  float r[16];
#pragma unroll
  // __fdividef (reciprocal + multiply, 2 ulp): the IEEE division's slow path is a subroutine call inside the epilogue,
  // and its mere presence cost the whole kernel 5-7 us at every row count (39.4 -> 34.4 us at 2 rows, 61.7 -> 54.6 at 256)
  for (int i = 0; i < 16; ++i) {
    const float gi = e.flip ? u[i] : g[i], ui = e.flip ? g[i] : u[i];
    r[i] = __fdividef(gi, 1.f + __expf(-gi)) * ui;
  }
  uint4* p = reinterpret_cast<uint4*>(e.out + (size_t)m * e.ld + j);
  p[0] = pack8(r);
  p[1] = pack8(r + 8);
}
__device__ __forceinline__ void epi16(const EpiQKVRope<bf16>& e, int m, int j, const float* a0, const float* a1,
                                      const EpiPre<EpiQKVRope<bf16>>& pre) {
  const int h = j / e.half, i = j % e.half;       // 16 indices stay inside one head (half is a multiple of 16)
  const int dh = 2 * e.half;
  float r0[16], r1[16];
  bf16* dst;
  if (h >= e.n_heads && e.seq_stride > 0 && e.row_seq[m] < 0) return;      // in-place layout: a row of no sequence has no cache slot
  if (h < e.n_heads + e.n_kv_heads) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 c = pre.c[q];                  // (cos, sin) of two consecutive frequencies
      r0[2 * q] = a0[2 * q] * c.x - a1[2 * q] * c.y;
      r1[2 * q] = a1[2 * q] * c.x + a0[2 * q] * c.y;
      r0[2 * q + 1] = a0[2 * q + 1] * c.z - a1[2 * q + 1] * c.w;
      r1[2 * q + 1] = a1[2 * q + 1] * c.z + a0[2 * q + 1] * c.w;
    }
    dst = (h < e.n_heads) ? e.q_out + (size_t)m * e.n_heads * dh + h * dh
                          : e.k_stage + e.kv_row(m) * e.n_kv_heads * dh + (h - e.n_heads) * dh;
  } else {
#pragma unroll
    for (int q = 0; q < 16; ++q) { r0[q] = a0[q]; r1[q] = a1[q]; }
    dst = e.v_stage + e.kv_row(m) * e.n_kv_heads * dh + (h - e.n_heads - e.n_kv_heads) * dh;
  }
  uint4* p0 = reinterpret_cast<uint4*>(dst + i);
  uint4* p1 = reinterpret_cast<uint4*>(dst + i + e.half);
  p0[0] = pack8(r0);
  p0[1] = pack8(r0 + 8);
  p1[0] = pack8(r1);
  p1[1] = pack8(r1 + 8);
}
__device__ __forceinline__ void epi16(const EpiQKVRope<bf16>& e, int m, int j, const float* a0, const float* a1) {
  EpiPre<EpiQKVRope<bf16>> pre;
  pre.load(e, m, j);
  epi16(e, m, j, a0, a1, pre);
}

// ---- host side ------------------------------------------------------------------------------------------------
typedef CUresult (*PFN_encodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct UmmaState {
  PFN_encodeTiled encode = nullptr;
  std::map<std::tuple<const void*, int, int, int, int, int>, CUtensorMap> cache4;
  std::map<std::tuple<const void*, size_t, int, int, int, int>, CUtensorMap> cache5;
  int max_smem = 0;
  int n_sm = 148;
  float* scratch = nullptr;        // split-K partial tiles (device), scratch_bytes long
  size_t scratch_bytes = 0;
  unsigned* counters = nullptr;    // split-K arrival counters (device), n_counters entries, zero between launches
  int n_counters = 0;
  int target_ctas = 0;             // 0 = one CTA per SM
  int max_stages = UM_MAX_STAGES;
  int pdl = 1;                     // launch with the programmatic-serialisation attribute
  int stream_cluster = 1;          // persistent kernel: K slices of a tile on one thread block cluster, reduced through DSMEM
  int max_clusters[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15};   // [c]: clusters of c one-per-SM CTAs that can be resident at once (queried at init)
  int stream_even = 0;             // persistent kernel: even shares over all SMs instead of equal K slices per tile
  int stream_bn = 0;               // its tile width (0 = automatic)
  int stream_bn_dual = 0;          // tile width of dual epilogues: 0 = automatic, 192 or 256
  int stream_exchange = 1;         // clusters of 2 exchange half tiles instead of publishing whole partial tiles
  int stream_exchange_rows = 64;   // ... from this many rows on
  int stream_atoms = 0;            // K atoms per stage: 0 = two when stream_min_stages2 such stages fit, else 1 or 2 as given
  int stream_min_stages2 = 3;
  int stream_split_copies = 0;     // a dual tile's weights by one copy per half and atom even where one copy can bring them all
  int pair_split = 0;              // its K slices (0 = automatic, 1 = never, 2 or 3 where they fit)
  int pair_bn = 0;                 // its tile width (0 = automatic)
  int pair_band = 0;               // its row groups per band (0 = automatic)
  std::set<const void*> smem_set;  // kernels whose shared-memory limit has been raised on this context's device
  std::string err;
};

// Raises a kernel's dynamic shared-memory limit once per library context: the limit belongs to the device (and the CUDA context)
// current at the call, so a flag per process would leave the kernel's launches on a second one to fail.
template <typename... KArgs>
cudaError_t umma_raise_smem(UmmaState& st, void (*kernel)(KArgs...)) {
  if (st.smem_set.count((const void*)kernel)) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, st.max_smem);
  if (e == cudaSuccess) st.smem_set.insert((const void*)kernel);
  return e;
}

inline int umma_init(UmmaState& st) {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
  if (e != cudaSuccess || fn == nullptr || qres != cudaDriverEntryPointSuccess) {
    st.err = "cuTensorMapEncodeTiled not available";
    return -1;
  }
  st.encode = (PFN_encodeTiled)fn;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&st.max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaDeviceGetAttribute(&st.n_sm, cudaDevAttrMultiProcessorCount, dev);
  return 0;
}

// bf16 tensor [rows, K] row-major seen as [K / 64 atoms][blocks of block_rows rows, block_stride rows apart][rows][64], so
// that one copy brings `atoms` K atoms of box_blocks x box_rows rows, each atom a [rows x 128 bytes] swizzled tile of its own
// behind the previous one (K atoms past the end are zero-filled).  Copies are issued by one thread at a cost that hardly
// depends on their size, so fewer and larger ones keep the producer ahead.  base: the first row (a rotary map starts at the
// head's first or second half).
inline CUresult umma_encode4(PFN_encodeTiled encode, CUtensorMap* m, const void* base, int block_rows, int block_stride, int blocks, int K,
                             int box_rows, int box_blocks, int atoms) {
  cuuint64_t dims[4] = {(cuuint64_t)UM_BK, (cuuint64_t)block_rows, (cuuint64_t)blocks, (cuuint64_t)(K / UM_BK)};
  cuuint64_t strides[3] = {(cuuint64_t)K * 2, (cuuint64_t)block_stride * K * 2, (cuuint64_t)UM_BK * 2};
  cuuint32_t box[4] = {(cuuint32_t)UM_BK, (cuuint32_t)box_rows, (cuuint32_t)box_blocks, (cuuint32_t)atoms};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}
inline const CUtensorMap* umma_map4(UmmaState& st, const void* base, int block_rows, int block_stride, int blocks, int K, int box_rows,
                                    int box_blocks, int atoms) {
  auto key = std::make_tuple(base, block_rows, block_stride, blocks, K, box_rows * 4096 + box_blocks * 16 + atoms);
  auto it = st.cache4.find(key);
  if (it != st.cache4.end()) return &it->second;
  if (st.cache4.size() > 4096) st.cache4.clear();
  CUtensorMap m;
  const CUresult r = umma_encode4(st.encode, &m, base, block_rows, block_stride, blocks, K, box_rows, box_blocks, atoms);
  if (r != CUDA_SUCCESS) {
    st.err = "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")";
    return nullptr;
  }
  return &st.cache4.emplace(key, m).first->second;
}

// Weight tiles of the row-major kernels: [K / 64 atoms][halves][blocks][rows][64], so that ONE copy brings both halves of a
// tile (gate / up rows, rotate-half partners) for `atoms` K atoms, laid out as the MMA wants them: per atom, the rows of the
// first half and then those of the second.
struct WeightView {
  const void* base;
  int rows, blocks, block_stride, halves;      // block_stride in rows
  size_t half_stride;                          // bytes between the halves
  int box_rows, box_blocks;                    // rows x blocks of a half tile
};
inline CUresult umma_encode5(PFN_encodeTiled encode, CUtensorMap* m, const WeightView& v, int K, int box_halves, int atoms) {
  cuuint64_t dims[5] = {(cuuint64_t)UM_BK, (cuuint64_t)v.rows, (cuuint64_t)v.blocks, (cuuint64_t)v.halves, (cuuint64_t)(K / UM_BK)};
  cuuint64_t strides[4] = {(cuuint64_t)K * 2, (cuuint64_t)v.block_stride * K * 2, (cuuint64_t)(v.halves > 1 ? v.half_stride : 16),
                           (cuuint64_t)UM_BK * 2};
  cuuint32_t box[5] = {(cuuint32_t)UM_BK, (cuuint32_t)v.box_rows, (cuuint32_t)v.box_blocks, (cuuint32_t)box_halves, (cuuint32_t)atoms};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(v.base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}
inline const CUtensorMap* umma_map5(UmmaState& st, const WeightView& v, int K, int atoms) {
  auto key = std::make_tuple(v.base, v.half_stride, v.rows, v.blocks, K, ((v.box_rows * 16 + v.box_blocks) * 4 + v.halves) * 16 + atoms);
  auto it = st.cache5.find(key);
  if (it != st.cache5.end()) return &it->second;
  if (st.cache5.size() > 4096) st.cache5.clear();
  CUtensorMap m;
  const CUresult r = umma_encode5(st.encode, &m, v, K, v.halves, atoms);
  if (r != CUDA_SUCCESS) {
    st.err = "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")";
    return nullptr;
  }
  return &st.cache5.emplace(key, m).first->second;
}

constexpr int UM_HEAD_BN = 256;
// More than 128 rows go to the pairs of SMs (gemm_pair.cuh).  With 129 to 256 rows (one row group) against the best kernels of
// one SM per tile, at 187 / 256 rows, us: 12288 x 4096 29 -> 26, 37 -> 27; 4096 x 4096 16.6 -> 14.9, 19.2 -> 15.1; 2 x 12288 SwiGLU
// 44.7 -> 46.3, 52.7 -> 48.0; 4096 x 12288 (three K slices) 30 -> 28.5; 3584 x 18944 38 -> 35.5; head 249 -> 199.  (The SwiGLU of
// 129 to 192 rows is the one launch that lost: 4 %, 43.3 -> 45.0 at 129.  Its MMAs span 256 rows whatever the row count, and its 128 tiles
// are two rounds of 74 pairs; 64-row MMAs for a second row tile on one SM, which it had, followed the rows more closely.)
inline bool umma_takes_pairs(int M) { return M > UM_BM; }
// The head's kernel and tile.  Its scores leave in fp32, so the rounding of the sums over K shows: the tensor core truncates at
// every step, and the error grows with the length of one accumulator's chain (scores of 4096 ids from K = 512, relative to
// 64 bits: 3.5e-6 in one chain, 1.7e-6 in two, 1.1e-6 in four).  A vocabulary of few tiles leaves tensor memory unused, one tile
// per pair: K then runs in four accumulators of 128 columns, or two of 256, which the epilogue adds in K order.
// Rows: more than 128 go to the pairs, as everywhere.  So do 9 to 128 with a short K: the streaming kernel would split the few
// tiles over its CTAs and sum them from global scratch (4096 ids, K 512: 49 us at 100 rows, 15.7 at 9, 13.0 at 4; pairs 15 to 16).
struct HeadShape { bool pairs; int bn, chains; };
inline HeadShape umma_head_shape(const UmmaState& st, int M, int vocab, int K) {
  const long rg = (M + 255) / 256, t256 = (vocab + 255) / 256 * rg, t128 = (vocab + 127) / 128 * rg, pairs = st.max_clusters[2];
  if (!(umma_takes_pairs(M) || (M > 8 && K <= 512 && t256 <= pairs))) return {false, UM_HEAD_BN, 1};
  if (t128 <= pairs) return {true, 128, 4};
  return {true, UM_HEAD_BN, t256 <= pairs ? 2 : 1};
}
// Partials per row the head GEMM leaves: one per vocabulary tile, or (k_gemm_pair) one per half tile.
inline int umma_head_tiles(const UmmaState& st, int M, int vocab, int K) {
  const HeadShape s = umma_head_shape(st, M, vocab, K);
  return (vocab + s.bn - 1) / s.bn * (s.pairs ? 2 : 1);
}

template <typename Epi> bool stream_can(const UmmaState& st, int M, int NP, int K, int bn);
template <typename Epi>
int pair_launch(UmmaState& st, cudaStream_t stream, const bf16* A, const bf16* W0, const bf16* W1, int M, int NP, int K,
                int n_rows_w, const Epi& epi, unsigned* status);
template <int BN, typename Epi>
int stream_launch(UmmaState& st, cudaStream_t stream, const bf16* A, const bf16* W0, const bf16* W1, int M, int NP, int K,
                  int n_rows_w, const Epi& epi, unsigned* status);

// More than 128 rows: pairs of SMs.  Else the streaming kernel (the K split follows from the tile count, see stream_launch)
// with this tile width, from measurements on the LLaDA and Dream layer shapes at 2 to 128 rows:
//  * the head 256;
//  * dual epilogues 256 columns (128 pairs), or 192 (96 pairs) where that makes one fuller wave: with 12288 pairs 128 tiles
//    instead of 96, i.e. a third more SMs pulling operands, and a quarter less shared-memory fill per CTA.  Only where no tile
//    would be split between CTAs (the split paths assume a power-of-two chunk count).  (The same idea for the rotary QKV
//    GEMM, 96-wide tiles that straddle heads, needs 16-row TMA boxes of 2 KB, and those cost far more than the fuller wave
//    gains: +0.7 ms per LLaDA-shaped pass.  Not kept.)
//  * plain and rotary ones 128, which needs no K split with 96 tiles.  With at most 32 rows a wide plain GEMM takes 256 (its partial
//    tiles are small, and half as many MMA instructions are issued), and so does a rotary one whose 128-wide tiles would be split
//    anyway; 96 whole tiles of 128 save the K slices' sum instead (12288 x 4096 in passes of 9 / 32 rows: 3.70 -> 3.58, 3.86 -> 3.68 ms).  K
//    then runs in as many accumulators as the 256-wide tiles would have slices, chunk by chunk in their order: one chain would be
//    longer than theirs, and the tensor core's error grows with the chain (see umma_head_shape); it was no faster (9 rows 3.58 and 3.58
//    ms).  The results are those of the 256-wide tiles to the bit.
//    A rotary half tile is whole head halves.
// A shape the kernel cannot take (none of a transformer layer's: it would need more than 4096 column tiles in a launch whose
// tiles are split between CTAs) is an error, not a fallback.
template <typename Epi>
int umma_gemm(UmmaState& st, cudaStream_t stream, const bf16* A, const bf16* W0, const bf16* W1, int M, int NP, int K,
              int n_rows_w, const Epi& epi, unsigned* status) {
  if (K % UM_BK) { st.err = "K must be a multiple of 64"; return -6; }
  if (Epi::kReduce ? umma_head_shape(st, M, NP, K).pairs : umma_takes_pairs(M))
    return pair_launch<Epi>(st, stream, A, W0, W1, M, NP, K, n_rows_w, epi, status);
  constexpr bool kRope = std::is_same<Epi, EpiQKVRope<bf16>>::value;
  const int cols = Epi::kDual ? 2 * NP : NP;
  int bn = UM_HEAD_BN;
  if constexpr (kRope) {
    const long t128 = (cols + 127) / 128;
    bn = M <= 32 && (2 * t128 <= st.n_sm || t128 > st.n_sm) ? 256 : 128;
    if (st.stream_bn > 0) bn = st.stream_bn;
    if (bn / 2 < epi.half) bn = 2 * epi.half;
  } else if constexpr (Epi::kDual) {
    const long t192 = NP / 96, t256 = (NP + 127) / 128;
    const bool whole192 = NP % 96 == 0 && t192 <= st.n_sm && 2 * t192 > st.n_sm;
    if (whole192 && st.stream_bn_dual != 256 && !st.stream_even && st.target_ctas == 0 &&
        (st.stream_bn_dual == 192 || (t256 < t192 && t256 < st.n_sm)))
      bn = 192;
    else if (st.stream_bn > 0)
      bn = st.stream_bn;
  } else if constexpr (!Epi::kReduce) {
    bn = (M <= 32 && cols >= 8192) ? 256 : 128;
    if (st.stream_bn > 0) bn = st.stream_bn;
  }
  if (stream_can<Epi>(st, M, NP, K, bn)) {
    if (bn == 256) return stream_launch<256, Epi>(st, stream, A, W0, W1, M, NP, K, n_rows_w, epi, status);
    if constexpr (!Epi::kReduce) {
      if (bn == 128) return stream_launch<128, Epi>(st, stream, A, W0, W1, M, NP, K, n_rows_w, epi, status);
    }
    if constexpr (Epi::kDual && !kRope) {
      if (bn == 192) return stream_launch<192, Epi>(st, stream, A, W0, W1, M, NP, K, n_rows_w, epi, status);
    }
  }
  st.err = "the tcgen05 GEMM cannot take this shape";
  return -8;
}

}  // namespace lsp
