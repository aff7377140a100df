// LM head over the masked block positions, reduced in the same kernel to a
// softmax entropy and a Gumbel-max token per position (arXiv 2509.04185,
// Eqs. 6-7 and Algorithm 3 "compute probabilities"; EB input of Eq. 3).
//
// Kernels, in launch order on one stream:
//   compact_rows_kernel  (bf16 above 32 rows, or without CTA pairs) gathers the
//                        hidden rows of masked positions into
//                        a dense [rows_alloc, H] buffer and a row map; writes
//                        entropy = +inf / token = -1 for unmasked positions;
//   head_pair_kernel     (bf16) the LM head on CTA pairs (clusters of 2) with
//                        2-SM tcgen05 MMAs of M = 256: W and the masked
//                        hidden rows stream into shared-memory rings by TMA,
//                        rank 0 issues the MMAs into double-buffered fp32
//                        accumulators in tensor memory of both CTAs, and the
//                        epilogue warps reduce every logit to running
//                        statistics (max, sum of exponentials, entropy
//                        numerator, best Gumbel score and id) -- logits
//                        never reach HBM.  Two layouts, chosen from the
//                        live row count (see the kernel);
//   head_tc_kernel       (bf16) the same on single CTAs with 1-SM MMAs,
//                        swap-AB: 128 vocab rows of W are the M side (A,
//                        K-major), the masked hidden rows the N side (B,
//                        K-major); eight epilogue warps (two per TMEM lane
//                        quadrant, alternate 16-column chunks) reduce each
//                        logit column over the lanes.  The fallback where no
//                        cluster of two fits or the vocabulary is one tile;
//   head_f32_kernel      (fp32) the same over fp32 FMAs, finding the masked rows
//                        itself;
//   head_combine_kernel  merges the per-CTA statistics of each row into the
//                        entropy (nats), the token and, when asked for, the
//                        confidence max_v p_v = 1 / S.
//
// Both tcgen05 kernels also serve sbd_linear (y = x W^T, a template
// switch): the same main loop over all rows of x, an epilogue that stores
// the outputs; head_tc_kernel up to 160 rows, the pair kernel's rows layout
// above.  With K split over CTAs the fp32 partials of a tile add up inside a
// thread-block cluster (up to 160 rows, where clusters are as good a split), or
// go through the workspace to linear_reduce_kernel.
#include <math.h>

#include <type_traits>

#include "philox.cuh"
#include "sbd_internal.cuh"

namespace {

using namespace sbd_dev;

constexpr int kBM = 128;              // vocab rows per tile (MMA M)
constexpr int kBK = 64;               // hidden columns per TMA box (one 128-B swizzle atom)
constexpr int kABytes = kBM * kBK * 2;  // one W box
constexpr int kMaxStages = 16;
// A pipeline stage holds up to this many consecutive boxes along the hidden
// dimension (longer contiguous reads of every W row per stage), and the ring
// gets this many bytes of shared memory.  One CTA per SM; W is loaded with
// an L2 evict-first policy, the hidden rows (re-read by every CTA) in boxes
// of up to 128 rows.
constexpr int kMaxBoxes = 4;
constexpr int kRingBytes = 216 * 1024;
// Epilogue warps (warps 2, 3, ...): warp w reads the TMEM lanes of quadrant
// w % 4, and the two warps of one quadrant take alternate 16-column chunks.
constexpr int kEpiWarps = 8;
// Chunks of Gumbel noise an epilogue warp keeps in flight ahead of the one
// it reduces (loads from HBM take longer than the reduction of one chunk).
// Measured on GB300 with 2 to 6 chunks: 3 is best or within 0.5 us of it at
// every row count (15 rows 156.6 -> 155.0 us against 2; 512 rows -6 %); 6
// spills registers.
constexpr int kGAhead = 3;
constexpr int kEpiThreads = 32 * kEpiWarps;
// kLinear: K ranges of a cluster at most.
constexpr int kMaxRanges = 8;
// kLinear: whether K ranges of whole stages are about as long as each other.
constexpr bool even_ranges(int stages, int ranges) {
  return stages % ranges == 0 || stages >= 4 * ranges;
}
// Boxes of a stage at most for H columns in `ranges` K ranges: whole stages, and
// even ranges of them.  (Single boxes, for ranges alike to the box: 1024 -> 1024 at
// 1 to 160 rows 5.8-8.25 us, with stages of 4 boxes 5.3-8.0.)
int stage_boxes(int H, int ranges) {
  int b = kMaxBoxes;
  while (b > 1 && ((H / kBK) % b != 0 || !even_ranges(H / kBK / b, ranges))) b >>= 1;
  return b;
}
constexpr int kHeadThreads = 64 + kEpiThreads;   // warp 0 TMA, warp 1 MMA, then the epilogue
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// Shared-memory scratch of the tensor-core epilogue for `rows` hidden rows:
// per TMEM quadrant and row the running (m, S, T, best) and best id, then
// the row map; rounded to 1 KB.
__host__ __device__ constexpr int head_scratch_bytes(int rows) {
  return (4 * rows * (16 + 4) + rows * 4 + 1023) & ~1023;
}

// ------------------------------------------------------------ tcgen05 PTX
__device__ __forceinline__ void tc_alloc(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// D[tmem] (+)= A[smem desc] * B[smem desc]^T, bf16 inputs, fp32 accumulate.
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                            uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives once on the mbarrier when every tcgen05 op issued so far by this
// thread has completed.
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}
// 32 lanes x 16 consecutive 32-bit columns: thread t gets lane (base + t).
__device__ __forceinline__ void tc_ld_32x32b_x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tc_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Shared-memory matrix descriptor: K-major operand laid out by TMA with the
// 128-byte swizzle, rows 128 B apart, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t sw128_kmajor_desc(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);   // start address
  d |= (uint64_t)(16u >> 4) << 16;                 // leading byte offset (unused here)
  d |= (uint64_t)(1024u >> 4) << 32;               // stride byte offset: 8 rows x 128 B
  d |= (uint64_t)1u << 46;                         // descriptor version (tcgen05)
  d |= (uint64_t)2u << 61;                         // 128-byte swizzle
  return d;
}
// Instruction descriptor, kind::f16: bf16 A and B (K-major), fp32 D.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N) {
  return (1u << 4)                  // D format: f32
         | (1u << 7)                // A format: bf16
         | (1u << 10)               // B format: bf16
         | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ---- the CTA-pair (2-SM) forms.  Two CTAs of a cluster share one MMA of
// M = 256: each holds 128 rows of A and half of B's N rows (rank 0 the first
// half) at the same shared-memory offsets, and each gets its 128 rows of D
// in its own tensor memory.  Every tcgen05 instruction of a pair kernel uses
// cta_group::2; allocation and release are performed by one warp of each
// CTA together.
__device__ __forceinline__ void tc_alloc_pair(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
// Issued by one thread of the pair's rank-0 CTA.
__device__ __forceinline__ void tc_mma_bf16_pair(uint32_t d_tmem, uint64_t a_desc,
                                                 uint64_t b_desc, uint32_t idesc,
                                                 uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// One arrival on the mbarrier at this offset in every CTA of `cta_mask`
// once the pair's tcgen05 ops issued so far by this thread have completed.
__device__ __forceinline__ void tc_commit_pair(uint64_t* bar, uint16_t cta_mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(smem_u32(bar)),
      "h"(cta_mask)
      : "memory");
}
// TMA load into this CTA's shared memory whose completion is counted on an
// mbarrier of either CTA of the pair (bar: shared::cluster address).
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* map, uint32_t bar,
                                                 int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile"
      ".mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair_hint(void* dst, const CUtensorMap* map,
                                                      uint32_t bar, int c0, int c1,
                                                      uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile"
      ".mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void pair_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t pair_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// The shared::cluster address of this CTA's shared location `p` in the
// pair's rank-0 CTA.
__device__ __forceinline__ uint32_t at_rank0(const void* p) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar)
               : "memory");
}
// mbar_wait for a barrier that CTAs of the cluster arrive on.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, int* err) {
  const uint64_t t0 = globaltimer();
  for (uint32_t n = 0;; ++n) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((n & 63u) == 63u && globaltimer() - t0 > kWaitLimitNs) {
      record_error(err, SBD_DEVERR_TIMEOUT);
      return false;
    }
  }
}

// 16 bytes at the shared-memory address `addr` of CTA `rank` of the cluster.
__device__ __forceinline__ float4 ld_cta_v4(uint32_t addr, int rank) {
  uint32_t p;
  float4 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(p) : "r"(addr), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(p)
               : "memory");
  return v;
}

// Two values rounded to bf16 (nearest even), the first in the low half.
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// 32 bytes to global memory (a whole sector) in one store.
__device__ __forceinline__ void st_global_v8(void* p, const uint32_t (&v)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v[0]), "r"(v[1]),
               "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

// ------------------------------------------------------------ epilogue math
// Statistics of 16 logit columns over the 32 vocabulary rows of a warp
// (lane = row, vocabulary id v0 + lane; z the logits, g the Gumbel noise).
// Two passes: the column maxima of z log2(e) and of the Gumbel score
// z + tau g go through a transposed max butterfly (16 + 8 + 4 + 2 + 1 steps
// instead of 16 x 5); every lane then takes exp2 of its logits against the
// column maxima, and the sums of the exponentials and of their entropy terms
// go through the same butterfly with additions.  The best id is the lowest
// lane that reaches the column's best score (ties to the lowest id).  On
// return lanes 2c and 2c + 1 hold column c.
__device__ __forceinline__ RowStats chunk16_stats(const float (&z)[16], const float (&g)[16],
                                                  bool valid, float tau, int v0, int lane) {
  float s[16], sc[16], ms[16], mb[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    s[j] = valid ? z[j] * kLog2e : -INFINITY;
    sc[j] = valid ? fmaf(tau, g[j], z[j]) : -INFINITY;
    ms[j] = s[j];
    mb[j] = sc[j];
  }
#pragma unroll
  for (int lvl = 0; lvl < 4; ++lvl) {
    const int b = 16 >> lvl;
    const int half = 8 >> lvl;
    const bool upper = (lane & b) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float ks = upper ? ms[i + half] : ms[i];
      const float ss = upper ? ms[i] : ms[i + half];
      const float kb = upper ? mb[i + half] : mb[i];
      const float sb = upper ? mb[i] : mb[i + half];
      ms[i] = fmaxf(ks, __shfl_xor_sync(0xffffffffu, ss, b));
      mb[i] = fmaxf(kb, __shfl_xor_sync(0xffffffffu, sb, b));
    }
  }
  ms[0] = fmaxf(ms[0], __shfl_xor_sync(0xffffffffu, ms[0], 1));
  mb[0] = fmaxf(mb[0], __shfl_xor_sync(0xffffffffu, mb[0], 1));

  const int my_col = (lane >> 1) & 15;
  unsigned my_hits = 0u;
  float e[16], t[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const float m = __shfl_sync(0xffffffffu, ms[0], 2 * j);
    const float best = __shfl_sync(0xffffffffu, mb[0], 2 * j);
    const float d = s[j] - m;                  // <= 0 on valid lanes
    e[j] = valid ? ex2_ftz(d) : 0.f;
    t[j] = valid ? e[j] * d : 0.f;
    const unsigned hits = __ballot_sync(0xffffffffu, valid && sc[j] == best);
    if (my_col == j) my_hits = hits;
  }
#pragma unroll
  for (int lvl = 0; lvl < 4; ++lvl) {
    const int b = 16 >> lvl;
    const int half = 8 >> lvl;
    const bool upper = (lane & b) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float ke = upper ? e[i + half] : e[i];
      const float se = upper ? e[i] : e[i + half];
      const float kt = upper ? t[i + half] : t[i];
      const float st = upper ? t[i] : t[i + half];
      e[i] = ke + __shfl_xor_sync(0xffffffffu, se, b);
      t[i] = kt + __shfl_xor_sync(0xffffffffu, st, b);
    }
  }
  e[0] += __shfl_xor_sync(0xffffffffu, e[0], 1);
  t[0] += __shfl_xor_sync(0xffffffffu, t[0], 1);
  RowStats r;
  r.m = ms[0];
  r.S = e[0];
  r.T = t[0];
  r.best = mb[0];
  r.idx = my_hits ? v0 + __ffs(my_hits) - 1 : 0x7fffffff;
  return r;
}

struct StatsRef {
  float4* msTb;   // (m, S, T, best)
  int* idx;
};
__device__ __forceinline__ RowStats load_stats(const StatsRef& s, int i) {
  const float4 v = s.msTb[i];
  RowStats r;
  r.m = v.x;
  r.S = v.y;
  r.T = v.z;
  r.best = v.w;
  r.idx = s.idx[i];
  return r;
}
__device__ __forceinline__ void store_stats(const StatsRef& s, int i, const RowStats& r) {
  s.msTb[i] = make_float4(r.m, r.S, r.T, r.best);
  s.idx[i] = r.idx;
}

// ------------------------------------------------------------ compaction
__global__ void __launch_bounds__(256)
compact_rows_kernel(const uint8_t* __restrict__ hidden, const uint8_t* __restrict__ masked,
                    int BK, int row_bytes, uint8_t* __restrict__ hidden_c,
                    int32_t* __restrict__ row_map, int32_t* __restrict__ n_rows,
                    float* __restrict__ entropy, int32_t* __restrict__ token,
                    float* __restrict__ confidence) {
  grid_dependency_wait();
  grid_dependents_launch();
  const int row = blockIdx.x;
  const int t = threadIdx.x;
  // masked rows before `row`, and in total (BK <= 2 * blockDim.x)
  int before = 0, total = 0;
  for (int base = 0; base < BK; base += blockDim.x) {
    const int i = base + t;
    const bool mt = i < BK && masked[i] != 0;
    before += __syncthreads_count(mt && i < row);
    total += __syncthreads_count(mt);
  }
  int dst;
  bool copy = false;
  if (row < BK) {
    if (masked[row]) {
      dst = before;
      copy = true;
      if (t == 0) row_map[dst] = row;
    } else {
      dst = total + (row - before);
      if (t == 0) {
        entropy[row] = INFINITY;
        token[row] = -1;
        if (confidence) confidence[row] = 0.f;
      }
    }
  } else {
    dst = row;
  }
  const int n16 = row_bytes / 16;
  uint4* out = reinterpret_cast<uint4*>(hidden_c + (size_t)dst * row_bytes);
  const uint4* in = reinterpret_cast<const uint4*>(hidden + (size_t)row * row_bytes);
  for (int c = t; c < n16; c += blockDim.x) out[c] = copy ? in[c] : make_uint4(0, 0, 0, 0);
  if (row == 0 && t == 0) *n_rows = total;
}

// ------------------------------------------------------------ bf16 tcgen05
struct HeadArgs {
  const float* gumbel;   // noise rows [B*k, V] (noise from a buffer)
  uint32_t seed_lo, seed_hi, off_lo, off_hi;   // counter-based noise (kPhilox)
  const int32_t* row_map;
  const int32_t* n_rows;
  float4* part_msTb;     // [gridDim.x][rows_alloc]
  int32_t* part_idx;
  int* err;
  int V, H, rows_alloc, n_tiles;
  int ring_bytes;       // shared memory of the TMA ring (shaped in the kernel)
  uint32_t tmem_cols;
  float tau;
  int h_big;            // tallest hidden-row box encoded: 16, 64 or 128 rows
  __nv_bfloat16* y;     // kLinear: output [linear_rows, V]
  int linear_rows;      // kLinear: rows of x, all live
  int ksplit;           // kLinear: K ranges per output tile (1: y written directly)
  int w_rows;           // kLinear, pairs: W rows of a unit per CTA (a multiple of 16 up to 128)
  int k_cluster;        // kLinear: the ranges of a tile form one cluster and add up there
  int boxes;            // head_tc_kernel: 64-column boxes of a stage at most
  float* part_y;        // kLinear, ksplit > 1: fp32 partials [ksplit][linear_rows][V]
  // kInPlace: the flags of all n_flags rows, and what the compaction kernel
  // writes otherwise
  const uint8_t* masked;
  int n_flags;
  int prefetch;         // boxes of a CTA's first W rows brought into L2 early
  int32_t* row_map_out;
  int32_t* n_rows_out;
  float* entropy;
  int32_t* token;
  float* confidence;
};

// kPhilox: the Gumbel noise is generated in the epilogue (philox.cuh)
// instead of read from a [B*k, V] buffer.  kLinear: the plain product
// y = x W^T in bf16 (all rows of x live, no compaction, no noise); the
// epilogue stores the accumulators instead of reducing them.
template <bool kPhilox, bool kLinear>
__global__ void __launch_bounds__(kHeadThreads, 1)
head_tc_kernel(const __grid_constant__ CUtensorMap tmap_w,
               const __grid_constant__ CUtensorMap tmap_h,
               const __grid_constant__ CUtensorMap tmap_h64,
               const __grid_constant__ CUtensorMap tmap_h128, const HeadArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages];
  __shared__ __align__(8) uint64_t empty_bar[kMaxStages];
  __shared__ __align__(8) uint64_t tmem_full[2];
  __shared__ __align__(8) uint64_t tmem_empty[2];
  __shared__ uint32_t tmem_base_sh;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (sbase - smem_u32(smem_raw));

  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmap_w);
    tma_prefetch_desc(&tmap_h);
  }
  if (warp == 1) tc_alloc(&tmem_base_sh, a.tmem_cols);
  if constexpr (kLinear) {
    // Nothing says that the previous kernel on the stream did not write W, so
    // it is not read before that kernel is done; but its first boxes come into
    // L2 (which stays coherent) meanwhile.  With the early trigger below, the
    // four GEMMs of an 8B layer in turn took 90.5 -> 87.4 us at 16 rows,
    // 138.2 -> 128.6 at 160, 171.3 -> 167.0 at 512 (24 boxes: 89.3, 6: 88.1).
    if (warp == 0 && lane < 12) {
      const int kb = (a.H / kBK) * (int)(blockIdx.x % a.ksplit) / a.ksplit + lane;
      if (kb < a.H / kBK)
        tma_prefetch_l2_2d(&tmap_w, kb * kBK, (int)(blockIdx.x / a.ksplit) * kBM);
    }
  }
  // Everything below reads what the compaction kernel wrote.
  grid_dependency_wait();
  const int R = kLinear ? a.linear_rows : *a.n_rows;
  const int n_eff = R <= 16 ? 16 : ((R + 15) / 16) * 16;   // MMA N
  // Two accumulator buffers whenever two of the live width fit in the
  // tensor memory of the launch (half of it each), so that the epilogue of
  // one tile overlaps the MMAs of the next; one above 256 live rows.
  const int n_acc = 2 * n_eff <= (int)a.tmem_cols ? 2 : 1;
  const uint32_t acc_stride = a.tmem_cols / 2;
  // Epilogue scratch for the n_eff live rows first, then the ring, which
  // also gets what the allocation kept for the scratch of rows_alloc rows.
  uint8_t* ep = gbase;
  const int ep_bytes = head_scratch_bytes(n_eff);
  const int ring_bytes = a.ring_bytes + head_scratch_bytes(a.rows_alloc) - ep_bytes;
  uint8_t* ring = gbase + ep_bytes;
  const uint32_t rbase = sbase + ep_bytes;
  // Statistics of TMEM lane quadrant w (computed, not indexed from an array:
  // a per-thread array of the four would live in local memory).
  auto wstats = [&](int w) -> StatsRef {
    StatsRef r;
    r.msTb = reinterpret_cast<float4*>(ep) + w * n_eff;
    r.idx = reinterpret_cast<int*>(ep + (size_t)4 * n_eff * sizeof(float4)) + w * n_eff;
    return r;
  };
  int* rmap = reinterpret_cast<int*>(ep + (size_t)4 * n_eff * (sizeof(float4) + 4));
  // Ring shape from the actual row count: a stage holds `boxes` 64-column
  // boxes of W (16 KB each) and of the n_eff hidden rows.  Above two boxes,
  // as many as still leave 3 stages; two boxes as long as 2 stages fit;
  // then as many stages as fit.  (Two boxes in 2 stages measured faster
  // than one box in 4-5: 160 rows 233 -> 219 us, 256 rows 255 -> 249 us;
  // four boxes in 2 stages slower than two in 4 at 60 rows.)
  const int b_box = n_eff * kBK * 2;
  // kLinear at few rows: each output tile's K is cut into `ksplit` ranges,
  // and the (tile, range) units are spread over the CTAs
  const int ksplit = kLinear ? a.ksplit : 1;
  const int n_units = a.n_tiles * ksplit;
  // (a.boxes divides the columns.  Every division here is on the way to the first
  // load: with the ranges' part of this choice in the kernel, and fits() a
  // division, an 8B layer's four GEMMs took 86.6 us at 16 rows, 86.1 so, those of
  // a layer of 1024 and 2816 columns 26.8 and 24.6)
  auto fits = [&](int bx, int n_st) { return ring_bytes >= n_st * bx * (kABytes + b_box); };
  int boxes = kMaxBoxes;         // (4, 2 or 1, as the compiler sees: the loops over it are unrolled)
  while (boxes > 1 && (boxes > a.boxes || !fits(boxes, boxes > 2 ? 3 : 2))) boxes >>= 1;
  const int stage_bytes = boxes * (kABytes + b_box);     // [A boxes | B boxes]
  int stages = ring_bytes / stage_bytes;
  if (stages > kMaxStages) stages = kMaxStages;
  // Epilogue warps with a chunk of 16 columns to reduce, per TMEM quadrant;
  // the others skip the tile loop.
  const int n_chunks = (R + 15) / 16;
  const int n_sub = n_chunks < kEpiWarps / 4 ? (n_chunks > 0 ? n_chunks : 1) : kEpiWarps / 4;
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tmem_full[i], 1);
      mbar_init(&tmem_empty[i], 4 * n_sub);   // one arrival per working epilogue warp
    }
    fence_mbar_init();
  }
  if (warp >= 2) {
    const int te = threadIdx.x - 64;
    for (int i = te; i < n_eff; i += kEpiThreads) {
      rmap[i] = (!kLinear && i < R) ? a.row_map[i] : 0;
      for (int w = 0; w < 4; ++w) store_stats(wstats(w), i, rowstats_empty());
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_sh;
  // the stages of K range ks: kb_of(ks) .. kb_of(ks + 1) - 1
  const int num_st = a.H / (kBK * boxes);
  auto kb_of = [&](int ks) { return ksplit == 1 ? ks * num_st : ks * num_st / ksplit; };

  if (R > 0) {
    if (warp == 0) {
      // ------------------------------------------------ TMA producer
      if (lane == 0) {
        const uint64_t policy = l2_policy_evict_first();
        // the stage and its phase are counters, not quotients (see
        // head_pair_kernel's producer)
        int it = 0, s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x) {
          const int tile = u / ksplit, ks = u % ksplit;
          for (int kb = kb_of(ks); kb < kb_of(ks + 1); ++kb, ++it) {
            if (!mbar_wait(&empty_bar[s], ph ^ 1, a.err)) {
              ok = false;
              break;
            }
            uint8_t* st = ring + (size_t)s * stage_bytes;
            mbar_arrive_expect_tx(&full_bar[s], stage_bytes);
            for (int x = 0; x < boxes; ++x) {
              const int col = (kb * boxes + x) * kBK;
              tma_load_2d_hint(st + x * kABytes, &tmap_w, &full_bar[s], col, tile * kBM, policy);
              // the n_eff hidden rows the MMA reads, in the tallest boxes that
              // fit: these rows come from L2 for every vocabulary tile, where
              // the copy rate per SM grows with the box size
              uint8_t* hb = st + boxes * kABytes + x * b_box;
              int r0 = 0;
              if (a.h_big >= 128)
                for (; r0 + 128 <= n_eff; r0 += 128)
                  tma_load_2d(hb + r0 * 128, &tmap_h128, &full_bar[s], col, r0);
              if (a.h_big >= 64)
                for (; r0 + 64 <= n_eff; r0 += 64)
                  tma_load_2d(hb + r0 * 128, &tmap_h64, &full_bar[s], col, r0);
              for (; r0 < n_eff; r0 += 16) tma_load_2d(hb + r0 * 128, &tmap_h, &full_bar[s], col, r0);
            }
            if (++s == stages) {
              s = 0;
              ph ^= 1u;
            }
          }
        }
        // every copy is issued: the next kernel may come up and prefetch
        if constexpr (kLinear) grid_dependents_launch();
        // copies still in flight must land before the CTA exits
        for (int q = it - stages > 0 ? it - stages : 0; q < it; ++q)
          mbar_wait(&full_bar[q % stages], (q / stages) & 1, a.err);
      }
    } else if (warp == 1) {
      // ------------------------------------------------ MMA issuer
      if (lane == 0) {
        // N is split into MMAs of at most 256 columns
        const int n_hi = n_eff > 256 ? n_eff - 256 : 0;
        const uint32_t idesc_lo = idesc_bf16_f32(kBM, n_eff > 256 ? 256 : n_eff);
        const uint32_t idesc_hi = idesc_bf16_f32(kBM, n_hi > 0 ? n_hi : 16);
        int it = 0, local = 0, s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x, ++local) {
          const int acc = n_acc == 2 ? (local & 1) : 0;
          const uint32_t use = (uint32_t)(n_acc == 2 ? (local >> 1) : local);
          if (!mbar_wait(&tmem_empty[acc], (use & 1) ^ 1, a.err)) break;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + (uint32_t)acc * acc_stride;
          const int kb0 = kb_of(u % ksplit), kb1 = kb_of(u % ksplit + 1);
          for (int kb = kb0; kb < kb1; ++kb, ++it) {
            if (!mbar_wait(&full_bar[s], ph, a.err)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t st = rbase + (uint32_t)(s * stage_bytes);
            for (int x = 0; x < boxes; ++x) {
              const uint64_t adesc = sw128_kmajor_desc(st + x * kABytes);
              const uint64_t bdesc = sw128_kmajor_desc(st + boxes * kABytes + x * b_box);
#pragma unroll
              for (int kk = 0; kk < kBK / 16; ++kk) {
                const uint32_t accum = (kb != kb0 || x != 0 || kk != 0);
                tc_mma_bf16(d_tmem, adesc + 2 * kk, bdesc + 2 * kk, idesc_lo, accum);
                if (n_hi > 0)   // rows 256.. of B: 256 x 128 B further on, 256 columns on
                  tc_mma_bf16(d_tmem + 256, adesc + 2 * kk, bdesc + (256 * 128 >> 4) + 2 * kk,
                              idesc_hi, accum);
              }
            }
            tc_commit(&empty_bar[s]);
            if (++s == stages) {
              s = 0;
              ph ^= 1u;
            }
          }
          if (ok) tc_commit(&tmem_full[acc]);
        }
      }
    } else {
      // ------------------------------------------------ epilogue warps
      const int quad = warp & 3;               // TMEM lanes 32*quad .. 32*quad+31
      const StatsRef my_stats = wstats(quad);
      const int sub = (warp - 2) / 4;          // chunks sub, sub + n_sub, ... of 16 columns
      const bool noisy = kPhilox || (!kLinear && a.tau != 0.f && a.gumbel != nullptr);
      const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
      int local = 0;
      for (int u = blockIdx.x; sub < n_sub && u < n_units; u += gridDim.x, ++local) {
        const int tile = u / ksplit, ks = u % ksplit;
        const int acc = n_acc == 2 ? (local & 1) : 0;
        const uint32_t use = (uint32_t)(n_acc == 2 ? (local >> 1) : local);
        const int v0 = tile * kBM + quad * 32;
        const int v = v0 + lane;
        const bool valid = v < a.V;
        const uint32_t t_acc = tmem_base + lane_addr + (uint32_t)acc * acc_stride;
        // Gumbel noise of the first kGAhead chunks is loaded while the MMAs
        // run; each chunk's reduction then loads the chunk kGAhead further on.
        const int stride = 16 * n_sub;
        const int c_first = 16 * sub;
        float gq[kGAhead][16];
        if constexpr (!kPhilox) {
#pragma unroll
          for (int d = 0; d < kGAhead; ++d)
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int cn = c_first + d * stride + j;
              gq[d][j] = (noisy && valid && cn < R) ? __ldg(a.gumbel + (size_t)rmap[cn] * a.V + v) : 0.f;
            }
        }
        // the tcgen05.ld below is warp-collective: the warp goes on as a whole
        if (!__all_sync(0xffffffffu, mbar_wait(&tmem_full[acc], use & 1, a.err))) break;
        tc_fence_after();
        for (int c0 = c_first; c0 < R; c0 += stride) {
          float g[16];
          if constexpr (!kPhilox) {
#pragma unroll
            for (int j = 0; j < 16; ++j) g[j] = gq[0][j];
#pragma unroll
            for (int d = 0; d + 1 < kGAhead; ++d)
#pragma unroll
              for (int j = 0; j < 16; ++j) gq[d][j] = gq[d + 1][j];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int cn = c0 + kGAhead * stride + j;
              gq[kGAhead - 1][j] =
                  (noisy && valid && cn < R) ? __ldg(a.gumbel + (size_t)rmap[cn] * a.V + v) : 0.f;
            }
          } else if (noisy) {
            // The four lanes 4q..4q+3 share vocabulary ids 4(v div 4) ..
            // +3, i.e. one Philox counter per row: each lane computes the
            // calls of 4 of the chunk's 16 rows, and a 4 x 4 transpose inside
            // the group gives every lane word v mod 4 of all 16.
            const uint32_t vq = (uint32_t)v >> 2;
            const int i4 = lane & 3;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              const int rr = c0 + 4 * t + i4;
              const uint32_t n = rr < R ? (uint32_t)rmap[rr] : 0u;
              const uint4 x = sbd_philox::philox4x32_10(make_uint4(vq, n, a.off_lo, a.off_hi),
                                                        a.seed_lo, a.seed_hi);
              uint32_t b[4] = {0u, 0u, 0u, 0u};
#pragma unroll
              for (int d = 0; d < 4; ++d) {
                // send word (i ^ d); receive word i of the call of row 4t + (i ^ d)
                const uint32_t send = sbd_philox::word_of(x, i4 ^ d);
                const uint32_t recv = d == 0 ? send : __shfl_xor_sync(0xffffffffu, send, d);
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) b[jj] = (jj == (i4 ^ d)) ? recv : b[jj];
              }
#pragma unroll
              for (int jj = 0; jj < 4; ++jj) g[4 * t + jj] = sbd_philox::gumbel_of_word(b[jj]);
            }
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) g[j] = 0.f;
          }
          uint32_t r[16];
          tc_ld_32x32b_x16(t_acc + (uint32_t)c0, r);
          tc_wait_ld();
          if constexpr (kLinear) {
            // y[c0 + j, v] (or its fp32 partial of K range ks): for each j the
            // warp's lanes store 32 consecutive v
            if (a.k_cluster) {
              // the range's partial, [row][vocabulary row of the tile], over
              // the ring: every stage was consumed before tmem_full
              float* pz = reinterpret_cast<float*>(ring) + c0 * kBM + quad * 32 + lane;
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (c0 + j < R) pz[j * kBM] = __uint_as_float(r[j]);
            } else if (valid) {
              if (ksplit == 1) {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                  if (c0 + j < R)
                    a.y[(size_t)(c0 + j) * a.V + v] = __float2bfloat16_rn(__uint_as_float(r[j]));
              } else {
                float* py = a.part_y + (size_t)ks * R * a.V;
#pragma unroll
                for (int j = 0; j < 16; ++j)
                  if (c0 + j < R) py[(size_t)(c0 + j) * a.V + v] = __uint_as_float(r[j]);
              }
            }
          } else {
            float z[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] = __uint_as_float(r[j]);
            const RowStats st = chunk16_stats(z, g, valid, a.tau, v0, lane);
            const int col = c0 + ((lane >> 1) & 15);
            if ((lane & 1) == 0 && col < R)
              store_stats(my_stats, col, rowstats_merge(load_stats(my_stats, col), st));
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tmem_empty[acc]);
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
      const int te = threadIdx.x - 64;
      if constexpr (!kLinear) {
        for (int col = te; col < R; col += kEpiThreads) {
          RowStats s = load_stats(wstats(0), col);
          for (int w = 1; w < 4; ++w) s = rowstats_merge(s, load_stats(wstats(w), col));
          const size_t o = (size_t)blockIdx.x * a.rows_alloc + col;
          a.part_msTb[o] = make_float4(s.m, s.S, s.T, s.best);
          a.part_idx[o] = s.idx;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tc_dealloc(tmem_base, a.tmem_cols);
  }
  if constexpr (kLinear) {
    if (a.k_cluster) {
      // y = the sum over the cluster's ranges, in range order: CTA `ks` takes
      // rows ks, ks + ksplit, ..., a warp a row, a lane 4 outputs.  The second
      // barrier keeps every CTA's partial alive until the others have read it.
      pair_sync();
      const int ks = (int)(blockIdx.x % ksplit), v0 = (int)(blockIdx.x / ksplit) * kBM + 4 * lane;
      const uint32_t zb = smem_u32(ring) + 16u * lane;
      const bool vec = a.V % 4 == 0 && v0 + 4 <= a.V;
      for (int r = ks + ksplit * warp; r < R; r += ksplit * (kHeadThreads / 32)) {
        float4 v[kMaxRanges];
#pragma unroll
        for (int e = 0; e < kMaxRanges; ++e)
          if (e < ksplit) v[e] = ld_cta_v4(zb + (uint32_t)(r * kBM * 4), e);
        float4 acc = v[0];
#pragma unroll
        for (int e = 1; e < kMaxRanges; ++e)
          if (e < ksplit) {
            acc.x += v[e].x;
            acc.y += v[e].y;
            acc.z += v[e].z;
            acc.w += v[e].w;
          }
        __nv_bfloat16* y = a.y + (size_t)r * a.V + v0;
        if (vec) {
          uint2 w;
          w.x = pack_bf16x2(acc.x, acc.y);
          w.y = pack_bf16x2(acc.z, acc.w);
          *reinterpret_cast<uint2*>(y) = w;
        } else {
          const float o[4] = {acc.x, acc.y, acc.z, acc.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (v0 + j < a.V) y[j] = __float2bfloat16_rn(o[j]);
        }
      }
      pair_sync();
    }
  }
}

// ------------------------------------------------------------ bf16 tcgen05, CTA pairs
// head_pair_kernel: the LM head on CTA pairs (clusters of 2) running 2-SM
// MMAs of M = 256.  A unit of work is a pair tile of 256 vocabulary rows
// (128 W rows in each CTA).  Both CTAs' copies complete on rank 0's full
// barriers; rank 0's thread issues the MMAs and commits them to the barriers
// of both CTAs; the epilogue warps of rank 1 release an accumulator on rank
// 0's barrier.  Two layouts, chosen from the live row count R:
//  - Rows mode (R > kPairVocabLanesMax = 160): the hidden rows are the A side
//    (TMEM lane = hidden row, 128 per CTA) and W the B side (N = 256), so
//    that each CTA's accumulator holds its rows' logits over all 256 ids of
//    the tile.  Each epilogue thread owns one row and folds its logits into
//    running statistics in registers, with no exchange between lanes; the
//    two warps of a lane quadrant take alternate 16-column chunks and merge
//    at the end.  Above 256 live rows there are two row groups; the pairs
//    take one group each, and the two pairs of a tile run at the same time
//    (W's lines come from L2 for the second).
//  - Vocabulary mode (R <= kPairVocabLanesMax): as in head_tc_kernel, W is
//    the A side (TMEM lane = vocabulary row) and the live rows the B side
//    (N = R padded to 32, half of them in each CTA), with the column
//    reductions over lanes.  The MMA's work then grows with R instead of
//    being fixed at 256 rows.
// Measured on GB300: a 2-SM MMA of N = 256 takes ~65 ns, the same rate per
// SM as a 1-SM MMA; what the pair gains is that each SM reads half of the
// hidden rows from L2 (the B operand is split between the two CTAs).  The
// vocabulary layout's time grows with its padded N (when the threshold was
// set: 131 live rows 192 us, 160 rows 198 us, 161-192 rows, padded to 192,
// 222 us) while the rows layout took ~212 us anywhere from 129 to 256 rows;
// re-checked on the current kernel, the rows layout is still slower at 131
// rows (190.0 against 187.5 us).  Below that the rows layout's fixed
// 256-row MMAs also cost power (it ran at ~1750 MHz and ~950 W at 60 live
// rows, against 2070 MHz and ~450 W for head_tc_kernel) and lost to it.
constexpr int kPairRows = 128;                 // hidden rows of one CTA per unit (M / 2)
constexpr int kPairVocabLanesMax = 160;        // live rows up to which the vocabulary layout runs
constexpr int kPrefetchAtOnce = 4;             // in place: boxes of W brought into L2 unasked

// One 16-column chunk of a row's logits z (vocabulary ids v0 .. v0 + 15, valid
// below V; kFull: all of them are) folded into the running maximum and sums;
// returns the chunk's maximum of z log2(e) (-inf when no id is valid).
template <bool kFull>
__device__ __forceinline__ float fold_sums16(RowStats& st, const float (&z)[16], int v0, int V) {
  float y[16];
  float mc = -INFINITY;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    y[j] = kFull || v0 + j < V ? z[j] * kLog2e : -INFINITY;
    mc = fmaxf(mc, y[j]);
  }
  if (mc == -INFINITY) return mc;               // no valid id in this chunk
  const float m_new = fmaxf(st.m, mc);
  float s_add = 0.f, t_add = 0.f;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    // invalid ids: 2^-1000 flushes to 0, and 0 * -1000 adds nothing to T
    const float d = kFull || v0 + j < V ? y[j] - m_new : -1000.f;
    const float e = ex2_ftz(d);
    s_add += e;
    t_add = fmaf(e, d, t_add);
  }
  if (st.S > 0.f) {
    // rescale the old sums to the new maximum: T' = 2^dm (T + dm S)
    const float dm = st.m - m_new;
    const float alpha = ex2_ftz(dm);
    st.T = fmaf(alpha, fmaf(dm, st.S, st.T), t_add);
    st.S = fmaf(alpha, st.S, s_add);
  } else {
    st.T = t_add;
    st.S = s_add;
  }
  st.m = m_new;
  return mc;
}

// The chunk's best Gumbel score z + tau g, noise g read.
template <bool kFull>
__device__ __forceinline__ void fold_scores16(RowStats& st, const float (&z)[16],
                                              const float (&g)[16], float tau, int v0, int V) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    // ids ascend within the chunk: a strict > keeps the lowest id on ties
    const float sc = fmaf(tau, g[j], z[j]);
    if ((kFull || v0 + j < V) && sc > st.best) {
      st.best = sc;
      st.idx = v0 + j;
    }
  }
}

// The same with the noise still in its random words x[j] (tau > 0; mc the
// chunk's maximum of z log2(e)).  A score beats st.best only if its noise
// exceeds d = (best - max z) / tau; the noise of 1 - u = (m + 1/2) 2^-23, with
// m = ~x >> 9, does so only if 1 - u < -ln u < exp(-d), so one compare a word
// against a bound shared by the chunk rules out nearly all of them without a
// logarithm: a row sees a new best about ln n times in n ids.  The others are
// scored exactly, in ascending order, so the winner is that of scoring every
// id.  d is lowered by more than the roundings of the noise (1e-5 here), the
// score (2^-24 of it) and this bound, and every comparison that is not
// decided (infinite or NaN d) falls on the exact side or cannot win.
// Per call at V = 128256, H = 4096 (bursts), two logarithms a logit against
// this: 200 rows 227 -> 205 us, 256 rows 225 -> 210, 320 rows 435 -> 385, 512
// rows 460 -> 380 (the noise buffer: 203, 209, 346, 351); V = 151936, 512
// rows, under the power cap 480 -> 441-453.  The rule by x_top and a lane's
// own order took 278 rows of 1280, 31919 ids from 67 to 57 us (98 without the
// rule when the logits spread 8 times as far; 69 scoring every id), 323 rows
// of 832, 80096 ids from 111 to 98 (182; 129).  Most of the rest are the generator's
// rounds.  (Round keys from the host made no difference.)
template <bool kFull>
__device__ __forceinline__ void fold_words16(RowStats& st, const float (&z)[16],
                                             const uint32_t (&x)[16], float mc, float tau,
                                             float inv_tau, int v0, int V) {
  const float z_max = fmaf(fabsf(mc), 1e-6f, mc * kLn2);
  const float d = (st.best - z_max) * inv_tau;
  const float eps =
      fmaf(fabsf(d), 1e-5f, fmaf(fabsf(st.best) + fabsf(z_max), 1e-6f * inv_tau, 5e-5f));
  // exp(-(d - eps)) 2^23, rounded up; above 2^23 every word qualifies
  const float bound = fmaf(ex2_ftz((eps - d) * kLog2e), 8388608.f * 1.0001f, 1.f);
  const uint32_t t = bound < 8388608.f ? (uint32_t)bound + 1u : 8388608u;   // m < t qualifies
  const uint32_t x_min = 0u - (t << 9);          // ~x >> 9 < t; 0 when t = 2^23
  uint32_t x_top = 0u;
#pragma unroll
  for (int j = 0; j < 16; ++j) x_top = max(x_top, x[j]);
  if (x_top < x_min) return;
  // A chunk with a new largest logit passes every word; but no noise of the
  // chunk is above that of x_top, which rules out the ids whose logit is too
  // far below the best even with it (the same slack).
  const float g_top = sbd_philox::gumbel_of_word(x_top);
  const float z_min =
      st.best - tau * g_top -
      fmaf(tau, fmaf(fabsf(g_top), 2e-5f, 1e-4f), 1e-6f * (fabsf(st.best) + fabsf(z_max)));
  // The lanes (rows) find theirs at different j: each takes its own next one,
  // so that a warp goes round as often as its busiest row has any, not once
  // for every j that some row has.
  uint32_t cand = 0u;
#pragma unroll
  for (int j = 0; j < 16; ++j)
    cand |= x[j] >= x_min && !(z[j] < z_min) && (kFull || v0 + j < V) ? 1u << j : 0u;
  while (cand != 0u) {
    const int j = __ffs(cand) - 1;
    cand &= cand - 1u;
    uint32_t xs[8];
    float zs[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      xs[i] = j & 8 ? x[i + 8] : x[i];
      zs[i] = j & 8 ? z[i + 8] : z[i];
    }
#pragma unroll
    for (int w = 4; w > 0; w >>= 1)
#pragma unroll
      for (int i = 0; i < w; ++i) {
        xs[i] = j & w ? xs[i + w] : xs[i];
        zs[i] = j & w ? zs[i + w] : zs[i];
      }
    const float sc = fmaf(tau, sbd_philox::gumbel_of_word(xs[0]), zs[0]);
    if (sc > st.best) {
      st.best = sc;
      st.idx = v0 + j;
    }
  }
}

// kLinear: sbd_linear's product y = x W^T (all rows of x live, no noise),
// always in the rows layout, the epilogue storing each row's outputs; with
// a.ksplit > 1 each (pair tile, K range) is a unit and the epilogue stores
// fp32 partials for linear_reduce_kernel.
// kInPlace: up to kInPlaceRows rows, read where they are (no compaction): all of
// them go through the MMAs, which take that many columns in any case, unless
// none is masked.  (An instance of its own: the same switch at run time cost
// the compacted calls 0.2-0.5 us.)
// kFew: at most kFewRows rows, so never the rows layout.
template <bool kPhilox, bool kLinear, bool kInPlace = false, bool kFew = kInPlace>
__global__ void __launch_bounds__(kHeadThreads, 1)
head_pair_kernel(const __grid_constant__ CUtensorMap tmap_w,
                 const __grid_constant__ CUtensorMap tmap_h,
                 const __grid_constant__ CUtensorMap tmap_h64,
                 const __grid_constant__ CUtensorMap tmap_h128, const HeadArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages];
  __shared__ __align__(8) uint64_t empty_bar[kMaxStages];
  __shared__ __align__(8) uint64_t tmem_full[2];
  __shared__ __align__(8) uint64_t tmem_empty[2];
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ float4 half_msTb[kPairRows];   // the second warp of each quadrant's row statistics
  __shared__ int half_idx[kPairRows];
  static_assert(!(kPhilox && kLinear), "the linear form has no noise");

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (sbase - smem_u32(smem_raw));
  const int rank = (int)pair_rank();
  const int pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);

  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmap_w);
    tma_prefetch_desc(&tmap_h);
  }
  // W rows of a unit in each CTA (head: 128)
  const int w_rows = kLinear ? a.w_rows : kBM;
  if constexpr (kLinear) {
    // W does not depend on the previous kernel in practice, but nothing says
    // so: its first boxes are brought into L2 only, which stays coherent, while
    // that kernel finishes (see head_tc_kernel)
    if (warp == 0 && lane < 6) {
      const int tk = pair / (a.linear_rows > 2 * kPairRows ? 2 : 1);
      const int kb = (a.H / kBK) / a.ksplit * (tk % a.ksplit) + lane;
      if (kb < a.H / kBK)
        tma_prefetch_l2_2d(&tmap_w, kb * kBK, (2 * (tk / a.ksplit) + rank) * w_rows);
    }
  }
  if constexpr (kInPlace) {
    // (as above: L2 only.)  With no row masked W is not read: the greater part
    // follows once a flag is seen, on a warp that has nothing else to do yet.  The
    // flags may still change before the wait below; here they only decide about
    // the prefetch, and the load stays out of L1.
    if (warp == 0 && lane < min(a.prefetch, kPrefetchAtOnce))
      tma_prefetch_l2_2d(&tmap_w, lane * kBK, (2 * pair + rank) * kBM);
    if (warp == 2 && a.prefetch > kPrefetchAtOnce) {
      uint32_t flag = 0;
      if (lane < a.n_flags)
        asm volatile("ld.relaxed.gpu.global.u8 %0, [%1];" : "=r"(flag) : "l"(a.masked + lane));
      if (__any_sync(0xffffffffu, flag != 0) && lane >= kPrefetchAtOnce && lane < a.prefetch)
        tma_prefetch_l2_2d(&tmap_w, lane * kBK, (2 * pair + rank) * kBM);
    }
  }
  // Everything below reads what the kernels before it wrote.
  grid_dependency_wait();
  uint32_t flags = 0;                              // kInPlace: the masked rows
  if constexpr (kInPlace)
    flags = __ballot_sync(0xffffffffu, lane < a.n_flags && a.masked[lane] != 0);
  const int R = kInPlace ? (flags != 0 ? a.n_flags : 0) : kLinear ? a.linear_rows : *a.n_rows;
  // The layout: hidden rows on the lanes above kPairVocabLanesMax live rows,
  // vocabulary rows on the lanes up to it.
  const bool rows_mode = kLinear || (!kFew && R > kPairVocabLanesMax);
  // Row groups of 2 x 128 rows (rows mode); each pair takes one group and
  // every per_group-th tile from its first one.
  const int n_groups = R > 2 * kPairRows ? 2 : 1;
  const int per_group = n_pairs / n_groups;
  const int grp = pair % n_groups;
  const bool working = R > 0 && pair < per_group * n_groups;
  const int t_first = pair / n_groups;
  // kLinear: K ranges per pair tile; a "tile" index below runs over
  // (pair tile, K range) pairs
  const int ksplit = kLinear ? a.ksplit : 1;
  const int n_tk = a.n_tiles * ksplit;
  // this CTA's hidden rows row0 .. row0 + 127 (live below R), and the peer's
  const int row0 = grp * 2 * kPairRows + rank * kPairRows;
  auto live_rows = [&](int r0) { return R - r0 < 0 ? 0 : (R - r0 > kPairRows ? kPairRows : R - r0); };
  const int live = live_rows(row0);
  const int live16 = (live + 15) / 16 * 16;                       // rows loaded
  const int peer16 = (live_rows(grp * 2 * kPairRows + (1 - rank) * kPairRows) + 15) / 16 * 16;
  // Ring: a stage holds `boxes` 64-column boxes of the hidden rows, then as
  // many of W (128 rows).  A hidden box takes the rows rank 0 of the group
  // loads (the larger share; the same layout in both CTAs): the MMA reads
  // 128 rows from its start, and the rows past the live ones come from the
  // next box or from W in the same stage, landed and only feeding the
  // accumulator lanes of rows that are not live.  So the ring holds as much
  // W as the live rows leave room for; as many boxes as still leave 3 stages.
  //
  // Vocabulary mode: the live rows padded to G (a multiple of 32), each CTA
  // loading G / 2 of them as its half of the B side; a stage holds `boxes`
  // boxes of W, then as many of the hidden rows.  The epilogue's running
  // statistics (per lane quadrant and row) and the row map sit in shared
  // memory before the ring.
  const int G = ((R > 0 ? R : 1) + 31) / 32 * 32;
  const int n_eff = R <= 16 ? 16 : (R + 15) / 16 * 16;
  const int ep_bytes = rows_mode ? 0 : head_scratch_bytes(n_eff);
  uint8_t* ep = gbase;
  uint8_t* ring = gbase + ep_bytes;
  const uint32_t rbase = sbase + (uint32_t)ep_bytes;
  const int ring_bytes = a.ring_bytes - ep_bytes;
  // (with fewer W rows a unit, a hidden box always takes 128 rows: the W boxes
  // behind the last one may not cover the 128 rows that the MMA reads)
  const int w_bytes = w_rows * kBK * 2;
  const int h_box = kLinear && w_rows < kBM ? kPairRows * kBK * 2
                    : rows_mode ? ((live_rows(grp * 2 * kPairRows) + 15) / 16 * 16) * kBK * 2
                                : (G / 2) * kBK * 2;
  // At least three stages.  (Two stages of longer W runs had measured 1-1.4 %
  // faster at 131 and 160 live rows while the control threads divided by
  // the stage count; with counters three are 1.5-2 % faster there.)
  const int min_stages = 3;
  int boxes = kMaxBoxes;
  while (boxes > 1 && ((a.H / kBK) % (boxes * ksplit) != 0 ||
                       ring_bytes / (boxes * (w_bytes + h_box)) < min_stages))
    boxes >>= 1;
  const int stage_bytes = boxes * (w_bytes + h_box);
  int stages = ring_bytes / stage_bytes;
  if (stages > kMaxStages) stages = kMaxStages;
  const int num_kb = a.H / (kBK * boxes) / ksplit;                 // stages per unit
  // offsets in a stage of W box x and hidden box x; the hidden rows loaded
  const int w_off0 = rows_mode ? boxes * h_box : 0;
  const int h_off0 = rows_mode ? 0 : boxes * w_bytes;
  const int h_first = rows_mode ? row0 : rank * (G / 2);
  const int h_count = rows_mode ? live16 : G / 2;
  // bytes landing per stage on rank 0's barrier: W and hidden rows of both CTAs
  const uint32_t tx_pair = rows_mode
      ? (uint32_t)boxes * (2u * (uint32_t)w_bytes + (uint32_t)(live16 + peer16) * 128u)
      : 2u * (uint32_t)stage_bytes;
  // vocabulary mode: statistics of TMEM lane quadrant w, and the row map
  auto wstats = [&](int w) -> StatsRef {
    StatsRef r;
    r.msTb = reinterpret_cast<float4*>(ep) + w * n_eff;
    r.idx = reinterpret_cast<int*>(ep + (size_t)4 * n_eff * sizeof(float4)) + w * n_eff;
    return r;
  };
  int* rmap = reinterpret_cast<int*>(ep + (size_t)4 * n_eff * (sizeof(float4) + 4));
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tmem_full[i], 1);
      mbar_init(&tmem_empty[i], 2 * kEpiWarps);   // every epilogue warp of both CTAs
    }
    mbar_init(&drain_bar, 1);
    fence_mbar_init();
  }
  if (!rows_mode && warp >= 2) {
    for (int i = threadIdx.x - 64; i < n_eff; i += kEpiThreads) {
      // (in place, a row that is not masked reads the first masked row's noise,
      // which costs no traffic; its statistics are not used)
      rmap[i] = i >= R ? 0 : !kInPlace ? a.row_map[i] : (flags >> i) & 1u ? i : __ffs(flags) - 1;
      for (int w = 0; w < 4; ++w) store_stats(wstats(w), i, rowstats_empty());
    }
  }
  if (kInPlace && blockIdx.x == 0 && warp == 1) {
    if (lane < a.n_flags) {
      const bool is_live = (flags >> lane) & 1u;
      a.row_map_out[lane] = is_live ? lane : -1;
      if (!is_live) {
        a.entropy[lane] = INFINITY;
        a.token[lane] = -1;
        if (a.confidence) a.confidence[lane] = 0.f;
      }
    }
    if (lane == 0) *a.n_rows_out = R;
  }
  // Both CTAs run and their barriers are initialised before either one
  // signals the other's; the pair then allocates its tensor memory.
  pair_sync();
  if (warp == 1) tc_alloc_pair(&tmem_base_sh, 512);
  tc_fence_before();
  // The producer warp only arrives: its copies need no tensor memory.  (In
  // the vocabulary layout with in-kernel noise 2-3 % faster than a full
  // barrier: 131 rows 203.1 -> 195.9 us; elsewhere within 0.5 %.)
  if (warp == 0) asm volatile("bar.arrive 2, %0;" ::"n"(kHeadThreads) : "memory");
  else asm volatile("bar.sync 2, %0;" ::"n"(kHeadThreads) : "memory");
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_sh;

  if (working) {
    if (warp == 0) {
      // ------------------------------------------------ TMA producer
      if (lane == 0) {
        // W is read once: evict-first, except where two row groups share it
        const bool w_hint = n_groups == 1;
        const uint64_t policy = l2_policy_evict_first();
        // This thread shares an SM sub-partition with two busy epilogue warps
        // and issues every copy, so its loop keeps little arithmetic per
        // stage: the stage and its phase are counters, not quotients by the
        // (run-time) stage count.  On GB300 that took the 60-row call from
        // 174.5 to 166.6 us and the 512-row one 8 % down (same for the MMA
        // thread below).
        int it = 0, s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int tk = t_first; ok && tk < n_tk; tk += per_group) {
          const int t = tk / ksplit, kb0 = (tk % ksplit) * num_kb;
          const int w_row = (2 * t + rank) * w_rows;
          for (int kb = 0; kb < num_kb; ++kb, ++it) {
            if (!mbar_wait(&empty_bar[s], ph ^ 1, a.err)) {
              ok = false;
              break;
            }
            uint8_t* st = ring + (size_t)s * stage_bytes;
            if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], tx_pair);
            const uint32_t fb = at_rank0(&full_bar[s]);
            for (int x = 0; x < boxes; ++x) {
              const int col = ((kb0 + kb) * boxes + x) * kBK;
              uint8_t* wb = st + w_off0 + x * w_bytes;
              if (w_hint) tma_load_2d_pair_hint(wb, &tmap_w, fb, col, w_row, policy);
              else tma_load_2d_pair(wb, &tmap_w, fb, col, w_row);
              // the hidden rows in the tallest boxes that fit (from L2)
              uint8_t* hb = st + h_off0 + x * h_box;
              int r0 = 0;
              if (a.h_big >= 128)
                for (; r0 + 128 <= h_count; r0 += 128)
                  tma_load_2d_pair(hb + r0 * 128, &tmap_h128, fb, col, h_first + r0);
              if (a.h_big >= 64)
                for (; r0 + 64 <= h_count; r0 += 64)
                  tma_load_2d_pair(hb + r0 * 128, &tmap_h64, fb, col, h_first + r0);
              for (; r0 < h_count; r0 += 16)
                tma_load_2d_pair(hb + r0 * 128, &tmap_h, fb, col, h_first + r0);
            }
            if (++s == stages) {
              s = 0;
              ph ^= 1u;
            }
          }
        }
        // every copy is issued: the next kernel may come up and prefetch
        if constexpr (kLinear) grid_dependents_launch();
        // Copies still in flight must land before the CTA exits.  Rank 1
        // cannot wait on rank 0's full barriers: it waits until the MMAs
        // released its last stages, which they do only after they arrived.
        bool landed = true;
        for (int q = it - stages > 0 ? it - stages : 0; landed && q < it; ++q)
          landed = rank == 0 ? mbar_wait(&full_bar[q % stages], (q / stages) & 1, a.err)
                             : mbar_wait(&empty_bar[q % stages], (q / stages) & 1, a.err);
      }
    } else if (warp == 1) {
      // ------------------------------------------------ MMA issuer (rank 0)
      if (lane == 0 && rank == 0) {
        // rows mode: A = hidden rows, B = W (N = 256 vocabulary ids);
        // vocabulary mode: A = W, B = hidden rows (N = G)
        const uint32_t idesc = idesc_bf16_f32(2 * kPairRows, rows_mode ? 2 * w_rows : G);
        int it = 0, local = 0, s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int tk = t_first; ok && tk < n_tk; tk += per_group, ++local) {
          const int acc = local & 1;
          const uint32_t use = (uint32_t)(local >> 1);
          // both CTAs' epilogue warps release the accumulator here
          if (!mbar_wait_cluster(&tmem_empty[acc], (use & 1) ^ 1, a.err)) break;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + (uint32_t)acc * 256u;
          for (int kb = 0; kb < num_kb; ++kb, ++it) {
            if (!mbar_wait(&full_bar[s], ph, a.err)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t st = rbase + (uint32_t)(s * stage_bytes);
            for (int x = 0; x < boxes; ++x) {
              const uint32_t w_s = st + (uint32_t)(w_off0 + x * w_bytes);
              const uint32_t h_s = st + (uint32_t)(h_off0 + x * h_box);
              const uint64_t adesc = sw128_kmajor_desc(rows_mode ? h_s : w_s);
              const uint64_t bdesc = sw128_kmajor_desc(rows_mode ? w_s : h_s);
#pragma unroll
              for (int kk = 0; kk < kBK / 16; ++kk)
                tc_mma_bf16_pair(d_tmem, adesc + 2 * kk, bdesc + 2 * kk, idesc,
                                 (kb != 0 || x != 0 || kk != 0) ? 1u : 0u);
            }
            tc_commit_pair(&empty_bar[s], 0x3);
            if (++s == stages) {
              s = 0;
              ph ^= 1u;
            }
          }
          if (ok) tc_commit_pair(&tmem_full[acc], 0x3);
        }
        // the MMAs read both CTAs' shared memory: none may be in flight when
        // the pair leaves (this matters after a time-out only)
        tc_commit_pair(&drain_bar, 0x1);
        mbar_wait(&drain_bar, 0, a.err);
      }
    } else if (rows_mode) {
      // ------------------------------------------------ epilogue warps, rows mode
      const int quad = warp & 3;               // TMEM lanes 32*quad .. 32*quad+31
      const int sub = (warp - 2) >> 2;         // 16-column chunks sub, sub + 2, ... of a unit
      const int h = row0 + quad * 32 + lane;   // this thread's hidden row
      const bool row_live = h < R;
      const bool warp_live = __any_sync(0xffffffffu, row_live);
      const int n = !kLinear && row_live ? a.row_map[h] : 0;
      const bool noisy = kPhilox || (!kLinear && a.tau != 0.f && a.gumbel != nullptr);
      const float* grow = noisy && !kPhilox ? a.gumbel + (size_t)n * a.V : nullptr;
      // kLinear: 32-byte stores where base and row stride allow (each lane
      // writes its own row: 16-byte stores half-fill every sector), else 16-byte
      // ones where those are aligned (512 columns -> 1000 outputs, 161 to 512
      // rows: 14.7-15.0 us an element at a time, 7.6-8.1 so)
      const uintptr_t y_al = reinterpret_cast<uintptr_t>(a.y) | (uintptr_t)a.V * 2u;
      const uintptr_t p_al = reinterpret_cast<uintptr_t>(a.part_y) | (uintptr_t)a.V * 4u;
      const bool y_vec = (y_al & 31u) == 0, y_vec16 = (y_al & 15u) == 0;
      const bool p_vec = (p_al & 31u) == 0, p_vec16 = (p_al & 15u) == 0;
      const bool vec4 = ((reinterpret_cast<uintptr_t>(a.gumbel) | (uintptr_t)a.V * 4u) & 15u) == 0;
      const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
      constexpr int kChunks = 2 * kBM / 16 / 2;   // chunks of one warp per unit of 2 x 128 ids
      auto load_noise = [&](int v0, float (&g)[16]) {
        if (!(noisy && row_live)) {
#pragma unroll
          for (int j = 0; j < 16; ++j) g[j] = 0.f;
        } else if (vec4) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 q4 = v0 + 4 * i < a.V ? __ldg(reinterpret_cast<const float4*>(grow + v0) + i)
                                               : make_float4(0.f, 0.f, 0.f, 0.f);
            g[4 * i] = q4.x;
            g[4 * i + 1] = q4.y;
            g[4 * i + 2] = q4.z;
            g[4 * i + 3] = q4.w;
          }
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) g[j] = v0 + j < a.V ? __ldg(grow + v0 + j) : 0.f;
        }
      };
      RowStats st = rowstats_empty();
      const float inv_tau = 1.f / a.tau;
      int local = 0;
      for (int tk = t_first; tk < n_tk; tk += per_group, ++local) {
        const int t = tk / ksplit, ks = tk % ksplit;
        const int acc = local & 1;
        const uint32_t use = (uint32_t)(local >> 1);
        const int vt = t * 2 * w_rows;                  // first vocabulary id of the tile
        const uint32_t t_acc = tmem_base + lane_addr + (uint32_t)acc * 256u;
        // noise of the first kGAhead chunks is read while the MMAs run
        float gq[kGAhead][16];
        if constexpr (!kPhilox) {
#pragma unroll
          for (int d = 0; d < kGAhead; ++d) load_noise(vt + 16 * (sub + 2 * d), gq[d]);
        }
        // the tcgen05.ld below is warp-collective: the warp goes on as a whole
        if (!__all_sync(0xffffffffu, mbar_wait(&tmem_full[acc], use & 1, a.err))) break;
        tc_fence_after();
        if (warp_live) {
#pragma unroll 1
          for (int c = 0; c < (kLinear ? w_rows / 16 : kChunks); ++c) {
            const int col = 16 * (sub + 2 * c);
            float g[16];
            if constexpr (!kPhilox) {
#pragma unroll
              for (int j = 0; j < 16; ++j) g[j] = gq[0][j];
#pragma unroll
              for (int d = 0; d + 1 < kGAhead; ++d)
#pragma unroll
                for (int j = 0; j < 16; ++j) gq[d][j] = gq[d + 1][j];
              if (c + kGAhead < kChunks) load_noise(vt + col + 32 * kGAhead, gq[kGAhead - 1]);
            }
            uint32_t words[16];
            if constexpr (kPhilox) {
              // one call gives the words of ids 4q .. 4q + 3 (col is a multiple
              // of 16); made while the accumulators are on their way
              if (noisy && row_live) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  const uint4 x = sbd_philox::philox4x32_10(
                      make_uint4(((uint32_t)(vt + col) >> 2) + (uint32_t)i, (uint32_t)n, a.off_lo, a.off_hi),
                      a.seed_lo, a.seed_hi);
#pragma unroll
                  for (int w = 0; w < 4; ++w) words[4 * i + w] = sbd_philox::word_of(x, w);
                }
              }
            }
            uint32_t r[16];
            tc_ld_32x32b_x16(t_acc + (uint32_t)col, r);
            tc_wait_ld();
            if (row_live) {
              float z[16];
#pragma unroll
              for (int j = 0; j < 16; ++j) z[j] = __uint_as_float(r[j]);
              if constexpr (kLinear) {
                // y[h, vt + col + j], j < 16, below out_features (a.V), or
                // with K ranges the fp32 partial of range ks
                const int n0 = vt + col;
                if (ksplit > 1) {
                  float* pr = a.part_y + ((size_t)ks * R + h) * a.V + n0;
                  if (p_vec && n0 + 16 <= a.V) {
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                      const uint32_t q[8] = {r[8 * i],     r[8 * i + 1], r[8 * i + 2], r[8 * i + 3],
                                             r[8 * i + 4], r[8 * i + 5], r[8 * i + 6], r[8 * i + 7]};
                      st_global_v8(pr + 8 * i, q);
                    }
                  } else if (p_vec16 && n0 + 16 <= a.V) {
#pragma unroll
                    for (int j = 0; j < 16; j += 4)
                      *reinterpret_cast<float4*>(pr + j) = make_float4(z[j], z[j + 1], z[j + 2], z[j + 3]);
                  } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                      if (n0 + j < a.V) pr[j] = z[j];
                  }
                } else {
                  __nv_bfloat16* yr = a.y + (size_t)h * a.V + n0;
                  if (y_vec16 && n0 + 16 <= a.V) {
                    const uint32_t q[8] = {pack_bf16x2(z[0], z[1]),   pack_bf16x2(z[2], z[3]),
                                           pack_bf16x2(z[4], z[5]),   pack_bf16x2(z[6], z[7]),
                                           pack_bf16x2(z[8], z[9]),   pack_bf16x2(z[10], z[11]),
                                           pack_bf16x2(z[12], z[13]), pack_bf16x2(z[14], z[15])};
                    if (y_vec) {
                      st_global_v8(yr, q);
                    } else {
                      reinterpret_cast<uint4*>(yr)[0] = make_uint4(q[0], q[1], q[2], q[3]);
                      reinterpret_cast<uint4*>(yr)[1] = make_uint4(q[4], q[5], q[6], q[7]);
                    }
                  } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                      if (n0 + j < a.V) yr[j] = __float2bfloat16_rn(z[j]);
                  }
                }
              } else {
                const int v0 = vt + col;
                auto fold = [&](auto full) {
                  constexpr bool kFull = decltype(full)::value;
                  const float mc = fold_sums16<kFull>(st, z, v0, a.V);
                  // (in its first unit a row has new bests often: scoring all
                  // of it is cheaper there: 200 rows of 512, 8000 ids 31.0 ->
                  // 27.8 us, 512 rows 43.4 -> 40.2; a large vocabulary of 200
                  // rows 199.8 -> 202.1)
                  if (kPhilox && local > 0) {
                    if (mc != -INFINITY)
                      fold_words16<kFull>(st, z, words, mc, a.tau, inv_tau, v0, a.V);
                  } else {
                    if constexpr (kPhilox) {
#pragma unroll
                      for (int j = 0; j < 16; ++j)
                        g[j] = sbd_philox::gumbel_of_word(words[j]);
                    }
                    fold_scores16<kFull>(st, z, g, a.tau, v0, a.V);
                  }
                };
                if (v0 + 16 <= a.V) fold(std::true_type{});
                else fold(std::false_type{});
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (rank == 1) mbar_arrive_cluster(at_rank0(&tmem_empty[acc]));
          else mbar_arrive(&tmem_empty[acc]);
        }
      }
      // the two warps of a quadrant merge their halves of each row
      const int slot = quad * 32 + lane;
      if constexpr (!kLinear) {
      if (sub == 1) {
        half_msTb[slot] = make_float4(st.m, st.S, st.T, st.best);
        half_idx[slot] = st.idx;
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
      if (sub == 0 && row_live) {
        RowStats o;
        o.m = half_msTb[slot].x;
        o.S = half_msTb[slot].y;
        o.T = half_msTb[slot].z;
        o.best = half_msTb[slot].w;
        o.idx = half_idx[slot];
        st = rowstats_merge(st, o);
        const size_t off = (size_t)blockIdx.x * a.rows_alloc + h;
        a.part_msTb[off] = make_float4(st.m, st.S, st.T, st.best);
        a.part_idx[off] = st.idx;
      }
      }
    } else if constexpr (!kLinear) {
      // ------------------------------------------------ epilogue warps, vocabulary mode
      // As in head_tc_kernel: thread = vocabulary row (TMEM lane), chunks of
      // 16 hidden-row columns reduced over the warp (chunk16_stats) and
      // merged into the quadrant's statistics in shared memory.
      const int quad = warp & 3;
      const StatsRef my_stats = wstats(quad);
      const int sub = (warp - 2) >> 2;          // chunks sub, sub + 2, ... of 16 columns
      const bool noisy = kPhilox || (a.tau != 0.f && a.gumbel != nullptr);
      const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
      constexpr int kStride = 32;
      const int c_first = 16 * sub;
      int local = 0;
      for (int t = t_first; t < a.n_tiles; t += per_group, ++local) {
        const int acc = local & 1;
        const uint32_t use = (uint32_t)(local >> 1);
        const int v0 = (2 * t + rank) * kBM + quad * 32;
        const int v = v0 + lane;
        const bool valid = v < a.V;
        const uint32_t t_acc = tmem_base + lane_addr + (uint32_t)acc * 256u;
        // Gumbel noise of the first kGAhead chunks is loaded while the MMAs
        // run; each chunk's reduction then loads the chunk kGAhead further on.
        float gq[kGAhead][16];
        if constexpr (!kPhilox) {
#pragma unroll
          for (int d = 0; d < kGAhead; ++d)
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int cn = c_first + d * kStride + j;
              gq[d][j] = (noisy && valid && cn < R) ? __ldg(a.gumbel + (size_t)rmap[cn] * a.V + v) : 0.f;
            }
        }
        // the tcgen05.ld below is warp-collective: the warp goes on as a whole
        if (!__all_sync(0xffffffffu, mbar_wait(&tmem_full[acc], use & 1, a.err))) break;
        tc_fence_after();
        for (int c0 = c_first; c0 < R; c0 += kStride) {
          float g[16];
          if constexpr (!kPhilox) {
#pragma unroll
            for (int j = 0; j < 16; ++j) g[j] = gq[0][j];
#pragma unroll
            for (int d = 0; d + 1 < kGAhead; ++d)
#pragma unroll
              for (int j = 0; j < 16; ++j) gq[d][j] = gq[d + 1][j];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int cn = c0 + kGAhead * kStride + j;
              gq[kGAhead - 1][j] =
                  (noisy && valid && cn < R) ? __ldg(a.gumbel + (size_t)rmap[cn] * a.V + v) : 0.f;
            }
          } else if (noisy) {
            // lanes 4q .. 4q + 3 share one Philox counter per row: each lane
            // computes the calls of 4 of the chunk's 16 rows, and a 4 x 4
            // transpose inside the group gives every lane word v mod 4 of all 16
            const uint32_t vq = (uint32_t)v >> 2;
            const int i4 = lane & 3;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int rr = c0 + 4 * q + i4;
              const uint32_t n = rr < R ? (uint32_t)rmap[rr] : 0u;
              const uint4 x = sbd_philox::philox4x32_10(make_uint4(vq, n, a.off_lo, a.off_hi),
                                                        a.seed_lo, a.seed_hi);
              uint32_t b[4] = {0u, 0u, 0u, 0u};
#pragma unroll
              for (int d = 0; d < 4; ++d) {
                const uint32_t send = sbd_philox::word_of(x, i4 ^ d);
                const uint32_t recv = d == 0 ? send : __shfl_xor_sync(0xffffffffu, send, d);
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) b[jj] = (jj == (i4 ^ d)) ? recv : b[jj];
              }
#pragma unroll
              for (int jj = 0; jj < 4; ++jj) g[4 * q + jj] = sbd_philox::gumbel_of_word(b[jj]);
            }
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) g[j] = 0.f;
          }
          uint32_t r[16];
          tc_ld_32x32b_x16(t_acc + (uint32_t)c0, r);
          tc_wait_ld();
          float z[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) z[j] = __uint_as_float(r[j]);
          const RowStats cs = chunk16_stats(z, g, valid, a.tau, v0, lane);
          const int col = c0 + ((lane >> 1) & 15);
          if ((lane & 1) == 0 && col < R)
            store_stats(my_stats, col, rowstats_merge(load_stats(my_stats, col), cs));
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (rank == 1) mbar_arrive_cluster(at_rank0(&tmem_empty[acc]));
          else mbar_arrive(&tmem_empty[acc]);
        }
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
      for (int col = threadIdx.x - 64; col < R; col += kEpiThreads) {
        RowStats m4 = load_stats(wstats(0), col);
        for (int w = 1; w < 4; ++w) m4 = rowstats_merge(m4, load_stats(wstats(w), col));
        const size_t off = (size_t)blockIdx.x * a.rows_alloc + col;
        a.part_msTb[off] = make_float4(m4.m, m4.S, m4.T, m4.best);
        a.part_idx[off] = m4.idx;
      }
    }
  }
  // Partials of the live rows this CTA does not own (rows mode, or no work):
  // empty statistics (the combine merges every CTA's partial of every row).
  if (!kLinear && warp >= 2 && (rows_mode || !working)) {
    const RowStats e = rowstats_empty();
    for (int r = threadIdx.x - 64; r < R; r += kEpiThreads) {
      if (working && r >= row0 && r < row0 + kPairRows) continue;
      const size_t off = (size_t)blockIdx.x * a.rows_alloc + r;
      a.part_msTb[off] = make_float4(e.m, e.S, e.T, e.best);
      a.part_idx[off] = e.idx;
    }
  }
  tc_fence_before();
  __syncthreads();
  // neither CTA releases its tensor memory or leaves while the other may
  // still signal its barriers or read its shared memory
  pair_sync();
  if (warp == 1) {
    tc_fence_after();
    tc_dealloc_pair(tmem_base, 512);
  }
  pair_sync();
}

// ------------------------------------------------------------ fp32 SIMT
// One CTA per 128 vocabulary rows; the live hidden rows go in groups of up
// to 32.  W and the group's hidden rows stream through a ring of 4 shared-
// memory stages of 32 columns (cp.async), so each W element is read from
// global memory once per group.  A lane holds 8 vocabulary rows of TR hidden
// rows, a warp 128 x 2 TR logits over a share of every stage's columns: the 8
// warps split the columns (8 or 16 rows) or the columns and the rows (24 or
// 32 rows).  TR + 8 shared-memory reads feed 32 TR FMAs.  The partial logits
// meet in shared memory, and each warp reduces every eighth row over its 128
// ids (two passes: the maxima, then the sums against them).
//
// Bound: W's bytes up to ~16 rows, the FMAs above (128 per SM and cycle).
// The form before read both operands of every scalar FMA from shared memory
// with one stage and one thread per vocabulary row.  Per call with the merge,
// V = 32003, H = 2048 (262 MB of W: 39 us; 32 rows of FMAs: 52 us, 63 with the
// 251 tiles on 152 SMs): 1-8 rows 397-528 us before, 53 now; 9-16 rows 548-677
// and 72; 17-24 rows 700-835 and 105; 25-32 rows 853-985 and 128.5.  Shared
// memory returns 128 bytes a cycle to registers, broadcasts included: with 8
// rows x 4 ids a lane (12 reads for 128 FMAs) the reads bound it (32 rows 12 %
// slower).
constexpr int kF32HeadWarps = 8;
constexpr int kF32HeadThreads = 32 * kF32HeadWarps;
constexpr int kF32Cols = 32;
constexpr int kF32Stages = 4;
constexpr int kF32Rows = 32;                         // rows of a group
constexpr int kF32MaxRows = 512;                     // B k at most
constexpr int kF32StageFloats = (kBM + kF32Rows) * kF32Cols;
constexpr size_t kF32SmemBytes = sizeof(float) * kF32Stages * kF32StageFloats;
static_assert(kF32HeadWarps * 16 * kBM <= kF32Stages * kF32StageFloats, "the partial logits fit the ring");

// The 16-byte column c (of 8) of a staged W row, turned by the row, so that
// 8 consecutive rows' reads of one column fall into distinct banks.
__device__ __forceinline__ int f32_w_at(int row, int c) {
  return row * kF32Cols + (((c ^ row) & 7) << 2);
}

struct F32HeadTile {
  const float* w;          // W row v0
  const float* hidden;     // hidden [B k, H]
  const int* map;          // the group's hidden rows
  int H, v_left, rows;     // columns; vocabulary rows from v0; rows of the group
};

// Partial logits of the tile into ring as [warp][2 TR rows][kBM], up to 16
// rows (W's bytes bound it): a ring of 4 stages filled with cp.async, row by
// row; warp w takes 16-byte column w of every stage.
template <int TR>
__device__ __forceinline__ void f32_tile_ring(const F32HeadTile& t, float* ring) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_chunks = (t.H + kF32Cols - 1) / kF32Cols;
  const int c_ld = tid & 7, r_ld = tid >> 3;         // staged 16-byte column, first row
  const int vl = lane & 15;                          // ids vl + 16 j
  const int row0 = (lane >> 4) * TR;                 // rows row0 + r
  const float* h_row = t.hidden + (size_t)(r_ld < t.rows ? t.map[r_ld] : 0) * t.H;
  auto load = [&](int chunk) {
    float* ws = ring + (chunk % kF32Stages) * kF32StageFloats;
    float* hs = ws + kBM * kF32Cols;
    const int col = chunk * kF32Cols + 4 * c_ld;
    const bool in = col < t.H;
    const float* wp = t.w + (in ? col : 0);
#pragma unroll
    for (int i = 0; i < kBM * 8 / kF32HeadThreads; ++i) {
      const int row = r_ld + (kF32HeadThreads / 8) * i;
      const bool ok = in && row < t.v_left;
      cp_async16(ws + f32_w_at(row, c_ld), ok ? wp + (size_t)row * t.H : t.w, ok);
    }
    // (rows past the group's last are zeros, up to a multiple of 8)
    if (r_ld < ((t.rows + 7) & ~7))
      cp_async16(hs + r_ld * kF32Cols + 4 * c_ld, h_row + (in ? col : 0), in && r_ld < t.rows);
  };
#pragma unroll
  for (int c = 0; c < kF32Stages - 1; ++c) {
    if (c < n_chunks) load(c);
    cp_async_commit();
  }
  float acc[TR][8];
#pragma unroll
  for (int r = 0; r < TR; ++r)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[r][j] = 0.f;
  for (int chunk = 0; chunk < n_chunks; ++chunk) {
    cp_async_wait<kF32Stages - 2>();
    __syncthreads();                                 // chunk landed; chunk - 1 consumed
    if (chunk + kF32Stages - 1 < n_chunks) load(chunk + kF32Stages - 1);
    cp_async_commit();
    const float* ws = ring + (chunk % kF32Stages) * kF32StageFloats;
    const float* hs = ws + kBM * kF32Cols + row0 * kF32Cols;
    float4 x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      x[j] = *reinterpret_cast<const float4*>(ws + f32_w_at(vl + 16 * j, warp));
#pragma unroll
    for (int r = 0; r < TR; ++r) {
      const float4 hv = *reinterpret_cast<const float4*>(hs + r * kF32Cols + 4 * warp);
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[r][j] = dot4(hv, x[j], acc[r][j]);
    }
  }
  __syncthreads();                                   // every stage consumed
  float* zs = ring + (warp * 2 * TR + row0) * kBM + vl;
#pragma unroll
  for (int r = 0; r < TR; ++r)
#pragma unroll
    for (int j = 0; j < 8; ++j) zs[r * kBM + 16 * j] = acc[r][j];
  __syncthreads();
}

// The same as [column share][4 TR rows][kBM] above 16 rows (the FMAs bound
// it): warp w is row group w % 2 and takes 8 columns of every 32, share w / 2.
// The chunks are transposed on their way through registers into two buffers
// of shared memory ([column][id] and [column][row], 8-float groups turned by
// the column against bank conflicts of the stores): an
// operand register then always meets the same accumulators, which the
// register allocation can keep in the other bank.  With both operands read
// along the columns an FMA's operand and accumulator fell into one bank half
// of the time (dispatch stalls, 48 % of the FMA rate).
template <int TR>
__device__ __forceinline__ void f32_tile_cols(const F32HeadTile& t, float* ring) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_chunks = (t.H + kF32Cols - 1) / kF32Cols;
  const int c_ld = tid & 7, r_ld = tid >> 3;
  const int vl = 4 * (lane & 15);                    // ids vl .. + 3 and 64 + vl .. + 3
  const int row0 = (warp & 1) * 2 * TR + (lane >> 4) * TR;
  const int part = warp >> 1;
  constexpr int kIter = kBM * 8 / kF32HeadThreads;
  constexpr int kBuf = kF32Cols * (kBM + kF32Rows);  // floats of a buffer
  float4 wr[kIter], hr;
  const float* h_row = t.hidden + (size_t)(r_ld < t.rows ? t.map[r_ld] : 0) * t.H;
  auto fetch = [&](int chunk) {
    const int col = chunk * kF32Cols + 4 * c_ld;
    const bool in = col < t.H;
#pragma unroll
    for (int i = 0; i < kIter; ++i) {
      const int row = r_ld + (kF32HeadThreads / 8) * i;
      wr[i] = in && row < t.v_left
                  ? __ldg(reinterpret_cast<const float4*>(t.w + (size_t)row * t.H + col))
                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    hr = in && r_ld < t.rows ? *reinterpret_cast<const float4*>(h_row + col)
                             : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  const int turn_st = 8 * (c_ld >> 1);               // of columns 4 c_ld .. + 3
  auto put = [&](float* buf) {
#pragma unroll
    for (int i = 0; i < kIter; ++i) {
      float* d = buf + 4 * c_ld * kBM + ((r_ld + (kF32HeadThreads / 8) * i) ^ turn_st);
      d[0] = wr[i].x;
      d[kBM] = wr[i].y;
      d[2 * kBM] = wr[i].z;
      d[3 * kBM] = wr[i].w;
    }
    float* d = buf + kF32Cols * kBM + 4 * c_ld * kF32Rows + (r_ld ^ turn_st);
    d[0] = hr.x;
    d[kF32Rows] = hr.y;
    d[2 * kF32Rows] = hr.z;
    d[3 * kF32Rows] = hr.w;
  };
  float acc[TR][8];
#pragma unroll
  for (int r = 0; r < TR; ++r)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[r][j] = 0.f;
  // this thread's words of its share's columns 8 part + kk, relative to `at`
  const int at = 8 * part * kBM;
  const int x_at = vl ^ (8 * part);
  int h_at[TR / 2];
#pragma unroll
  for (int r = 0; r < TR; r += 2)
    h_at[r / 2] = kF32Cols * kBM - at + 8 * part * kF32Rows + ((row0 + r) ^ (8 * part));
  fetch(0);
  put(ring);
  if (n_chunks > 1) fetch(1);
  __syncthreads();
  for (int chunk = 0; chunk < n_chunks; ++chunk) {
    const float* buf = ring + (chunk & 1) * kBuf + at;
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
      const float4 x0 = *reinterpret_cast<const float4*>(buf + x_at + kk * kBM);
      const float4 x1 = *reinterpret_cast<const float4*>(buf + x_at + kk * kBM + 64);
      const float xs[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
      float h[TR];
#pragma unroll
      for (int r = 0; r < TR; r += 2) {
        const float2 v = *reinterpret_cast<const float2*>(buf + h_at[r / 2] + kk * kF32Rows);
        h[r] = v.x;
        h[r + 1] = v.y;
      }
#pragma unroll
      for (int r = 0; r < TR; ++r)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[r][j] = fmaf(h[r], xs[j], acc[r][j]);
    }
    if (chunk + 1 < n_chunks) {
      put(ring + ((chunk + 1) & 1) * kBuf);          // consumed before the last barrier
      if (chunk + 2 < n_chunks) fetch(chunk + 2);
    }
    __syncthreads();
  }
  float* zs = ring + (part * 4 * TR + row0) * kBM + vl;
#pragma unroll
  for (int r = 0; r < TR; ++r) {
    *reinterpret_cast<float4*>(zs + r * kBM) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
    *reinterpret_cast<float4*>(zs + r * kBM + 64) = make_float4(acc[r][4], acc[r][5], acc[r][6], acc[r][7]);
  }
  __syncthreads();
}

template <bool kPhilox>
__global__ void __launch_bounds__(kF32HeadThreads, 2)
head_f32_kernel(const float* __restrict__ hidden, const float* __restrict__ w,
                const float* __restrict__ gumbel, const uint8_t* __restrict__ masked, int BK,
                int32_t* __restrict__ row_map, int32_t* __restrict__ n_rows, float tau, int V,
                int H, int rows_alloc, float4* __restrict__ part_msTb,
                int32_t* __restrict__ part_idx, float* __restrict__ entropy,
                int32_t* __restrict__ token, float* __restrict__ confidence, uint4 philox_sk) {
  extern __shared__ __align__(16) float f32_smem[];
  // The masked rows in order: every CTA finds them for itself (B k <= 512
  // flags), the first one writes them out for the merge, and the unmasked
  // rows' results; the hidden rows are read where they are.  A kernel of its own
  // that did this and copied the rows, as for bf16, cost a launch: 1-3 rows of
  // hidden 256, 512 ids 8.8 -> 7.6 us, 32 rows of 2048, 32003 ids 3.5 us.
  __shared__ int rows_sh[kF32MaxRows], count_sh[kF32MaxRows / 32];
  grid_dependency_wait();
  for (int i0 = 0; i0 < kF32MaxRows; i0 += kF32HeadThreads) {
    const int i = i0 + threadIdx.x;
    const unsigned bal = __ballot_sync(0xffffffffu, i < BK && masked[i] != 0);
    if ((threadIdx.x & 31) == 0) count_sh[i / 32] = __popc(bal);
  }
  __syncthreads();
  int R = 0;
  for (int i0 = 0; i0 < kF32MaxRows; i0 += kF32HeadThreads) {
    const int i = i0 + threadIdx.x, ln = threadIdx.x & 31;
    // the counts of the groups of 32 before this one, and of all
    const int c = ln < kF32MaxRows / 32 ? count_sh[ln] : 0;
    const int before = __reduce_add_sync(0xffffffffu, ln < i / 32 ? c : 0);
    R = __reduce_add_sync(0xffffffffu, c);
    const bool live = i < BK && masked[i] != 0;
    const unsigned bal = __ballot_sync(0xffffffffu, live);
    const int at = before + __popc(bal & ((1u << ln) - 1u));
    if (live) rows_sh[at] = i;
    if (blockIdx.x == 0 && i < BK) {
      if (live) {
        row_map[at] = i;
      } else {
        entropy[i] = INFINITY;
        token[i] = -1;
        if (confidence) confidence[i] = 0.f;
      }
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *n_rows = R;
  __syncthreads();
  const int v0 = blockIdx.x * kBM;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool noisy = kPhilox || (tau != 0.f && gumbel != nullptr);
  const int vq = v0 + 4 * lane;                      // this lane's first id in the reduction

  for (int r0 = 0; r0 < R; r0 += kF32Rows) {
    const int nr = min(kF32Rows, R - r0);
    F32HeadTile t;
    t.w = w + (size_t)v0 * H;
    t.hidden = hidden;
    t.map = rows_sh + r0;
    t.H = H;
    t.v_left = V - v0;
    t.rows = nr;
    int zrows = 32, parts = 4;                       // [parts][zrows][kBM] partial logits
    if (nr <= 8) {
      f32_tile_ring<4>(t, f32_smem);
      zrows = 8, parts = 8;
    } else if (nr <= 16) {
      f32_tile_ring<8>(t, f32_smem);
      zrows = 16, parts = 8;
    } else if (nr <= 24) {
      f32_tile_cols<6>(t, f32_smem);
      zrows = 24;
    } else {
      f32_tile_cols<8>(t, f32_smem);
    }
    const float* zs = f32_smem;
    // noise of this warp's rows warp, warp + 8, ... of the group
    float g[kF32Rows / kF32HeadWarps][4];
#pragma unroll
    for (int i = 0; i < kF32Rows / kF32HeadWarps; ++i) {
      const int row = warp + kF32HeadWarps * i;
#pragma unroll
      for (int j = 0; j < 4; ++j) g[i][j] = 0.f;
      if (noisy && row < nr) {
        const int n = rows_sh[r0 + row];
        if constexpr (kPhilox) {
          // philox_sk = (seed low, seed high, offset low, offset high); the
          // lane's four ids are the four words of one call
          const uint4 x = sbd_philox::philox4x32_10(
              make_uint4((uint32_t)vq >> 2, (uint32_t)n, philox_sk.z, philox_sk.w), philox_sk.x,
              philox_sk.y);
#pragma unroll
          for (int j = 0; j < 4; ++j) g[i][j] = sbd_philox::gumbel_of_word(sbd_philox::word_of(x, j));
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (vq + j < V) g[i][j] = __ldg(gumbel + (size_t)n * V + vq + j);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kF32Rows / kF32HeadWarps; ++i) {
      const int row = warp + kF32HeadWarps * i;
      if (row >= nr) break;
      float z[4] = {0.f, 0.f, 0.f, 0.f};
      for (int p = 0; p < parts; ++p) {
        const float4 x = *reinterpret_cast<const float4*>(zs + (p * zrows + row) * kBM + 4 * lane);
        z[0] += x.x;
        z[1] += x.y;
        z[2] += x.z;
        z[3] += x.w;
      }
      float y[4], mx = -INFINITY, best = -INFINITY;
      int idx = vq;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool ok = vq + j < V;
        y[j] = z[j] * kLog2e;
        if (ok) mx = fmaxf(mx, y[j]);
        const float sc = fmaf(tau, g[i][j], z[j]);
        if (ok && sc > best) {                       // ids ascend: the lowest wins ties
          best = sc;
          idx = vq + j;
        }
      }
      const float m = warp_max(mx);
      const float wbest = warp_max(best);
      // the lowest lane that reaches the best score (lane 0's first id when
      // no score compares, i.e. every logit is NaN)
      const unsigned hits = __ballot_sync(0xffffffffu, vq < V && best == wbest);
      const int win = __shfl_sync(0xffffffffu, idx, hits ? __ffs(hits) - 1 : 0);
      float S = 0.f, T = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (vq + j < V && y[j] != -INFINITY) {       // m may be -inf, too
          const float d = y[j] - m;                  // <= 0
          const float e = exp2f(d);
          S += e;
          T = fmaf(e, d, T);
        }
      }
      S = warp_sum(S);
      T = warp_sum(T);
      if (lane == 0) {
        const size_t o = (size_t)blockIdx.x * rows_alloc + r0 + row;
        part_msTb[o] = make_float4(m, S, T, wbest);
        part_idx[o] = win;
      }
    }
    __syncthreads();                                 // the partial logits are read
  }
}

// ------------------------------------------------------------ combine
// One warp per masked row: merge the per-CTA statistics, then
// H = ln 2 * (log2 S - T / S)  (nats) and the winning token.  Latency-bound:
// the row count, the row map and up to 256 CTAs' statistics (8 per lane) are
// all requested before any of them is used.
__global__ void __launch_bounds__(128)
head_combine_kernel(const float4* __restrict__ part_msTb, const int32_t* __restrict__ part_idx,
                    int n_parts, int rows_alloc, const int32_t* __restrict__ row_map,
                    const int32_t* __restrict__ n_rows, float* __restrict__ entropy,
                    int32_t* __restrict__ token, float* __restrict__ confidence) {
  constexpr int kPerLane = 8;
  grid_dependency_wait();
  const int r = blockIdx.x * 4 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= rows_alloc) return;
  const int rows = *n_rows;
  const int row = row_map[r];        // read before the check: r < rows_alloc; -1: not masked
  RowStats s = rowstats_empty();
  for (int c0 = 0; c0 < n_parts; c0 += 32 * kPerLane) {
    float4 v[kPerLane];
    int id[kPerLane];
#pragma unroll
    for (int e = 0; e < kPerLane; ++e) {
      const int c = c0 + e * 32 + lane;
      if (c < n_parts) {
        v[e] = part_msTb[(size_t)c * rows_alloc + r];
        id[e] = part_idx[(size_t)c * rows_alloc + r];
      }
    }
#pragma unroll
    for (int e = 0; e < kPerLane; ++e) {
      if (c0 + e * 32 + lane < n_parts) {
        RowStats o;
        o.m = v[e].x;
        o.S = v[e].y;
        o.T = v[e].z;
        o.best = v[e].w;
        o.idx = id[e];
        s = rowstats_merge(s, o);
      }
    }
  }
  if (r >= rows || row < 0) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    RowStats t;
    t.m = __shfl_xor_sync(0xffffffffu, s.m, o);
    t.S = __shfl_xor_sync(0xffffffffu, s.S, o);
    t.T = __shfl_xor_sync(0xffffffffu, s.T, o);
    t.best = __shfl_xor_sync(0xffffffffu, s.best, o);
    t.idx = __shfl_xor_sync(0xffffffffu, s.idx, o);
    s = rowstats_merge(s, t);
  }
  if (lane == 0) {
    entropy[row] = kLn2 * (log2f(s.S) - s.T / s.S);
    token[row] = s.idx;
    // the largest probability is the max term's: 2^0 / S
    if (confidence) confidence[row] = 1.f / s.S;
  }
}

// ------------------------------------------------------------ workspace
struct HeadWs {
  uint8_t* hidden_c;       // the masked rows (bf16 only)
  int32_t* row_map;
  int32_t* n_rows;
  float4* part_msTb;
  int32_t* part_idx;
  size_t bytes;
};

HeadWs head_ws_layout(const sbd::HeadPlan& p, void* base) {
  HeadWs w;
  const uintptr_t c = reinterpret_cast<uintptr_t>(base);
  size_t off = 0;
  w.hidden_c = reinterpret_cast<uint8_t*>(c + off);
  // (fp32 reads its rows where they are, and keeps the size: the fixed scratch
  // of the no-allocation call takes the same shapes as ever)
  const size_t elem = p.bf16 ? 2 : 4;
  off = sbd::align_up(off + (size_t)p.rows_alloc * p.H * elem, 256);
  w.row_map = reinterpret_cast<int32_t*>(c + off);
  off = sbd::align_up(off + (size_t)p.rows_alloc * 4, 256);
  w.n_rows = reinterpret_cast<int32_t*>(c + off);
  off = sbd::align_up(off + 4, 256);
  w.part_msTb = reinterpret_cast<float4*>(c + off);
  off = sbd::align_up(off + (size_t)p.n_ctas * p.rows_alloc * sizeof(float4), 256);
  w.part_idx = reinterpret_cast<int32_t*>(c + off);
  off = sbd::align_up(off + (size_t)p.n_ctas * p.rows_alloc * 4, 256);
  w.bytes = off;
  return w;
}


// Shared memory of the ring: kRingBytes, within what a CTA can have next to
// the epilogue scratch.
int head_ring_bytes(int rows_alloc) {
  const int per_cta = 224 * 1024 - 1024 - 1024;
  int budget = kRingBytes;
  if (budget > per_cta - head_scratch_bytes(rows_alloc)) budget = per_cta - head_scratch_bytes(rows_alloc);
  return budget;
}

size_t head_smem_bytes(int rows_alloc) {
  return 1024 + (size_t)head_scratch_bytes(rows_alloc) + head_ring_bytes(rows_alloc);
}

// The LM head runs on CTA pairs (head_pair_kernel) from this many allocated
// rows, i.e. always (at 15 live rows it measured 161.1 us against 162.5 us
// for head_tc_kernel, which remains for a device that cannot hold a cluster
// of two and for a vocabulary of one tile); its shared memory is the ring
// alone.
constexpr int kPairMinRows = 16;
// Rows up to which the pair kernel takes the hidden rows where they are instead
// of compacted ones: its B side is padded to 32 rows in any case, so the rows
// that are not masked cost nothing in the MMAs, and a launch on the critical
// path goes.  16 rows of 4096, 128256 ids: 158.7 -> 156.7 us; 4 rows of 2048,
// 32000 ids: 30.5 -> 29.5; 32 rows, all masked, 160.8 -> 159.0, 3 of them
// 159.4 -> 158.9 (32000 ids, in-kernel noise: 32.8 -> 33.1).  Above 32 rows the
// padded N would grow with rows that are not masked.  (Compaction by TMA
// gather4 loads of the masked rows: 16 rows 158.5 -> 168.8, 64 rows 168 -> 246.)
constexpr int kInPlaceRows = 32;
// Rows up to which the compacted call with in-kernel noise has an instance
// without the rows layout, whose code had cost the vocabulary layout's noise
// registers: 14 of 60 rows of 1152, 135511 ids 61.7 -> 59.6 us, all 60 76.2 ->
// 73.9, 36 rows of 1024, 60000 ids 45.8 -> 44.1; 160 rows of 4096, 128256 ids
// 198.3 -> 199.7.  (Without noise 128 rows of 1024 41.5 -> 40.9 but 95 of 126
// rows of 960, 67692 ids 43.1 -> 44.0.)
constexpr int kFewRows = 128;
// Without the compaction kernel in between, the pair kernel comes up while the
// kernel before it (attention, in a step) still runs, and its first boxes of W
// are brought into L2 meanwhile; they are read from there once that kernel is
// done.  16 boxes: 32000 ids of 2048 29.3 -> 27.7 us (8 boxes 28.4; 32 27.8),
// 50304 of 1024 24.0 -> 23.2, 151936 of 4096 182.8 -> 180.7, 128256 158.3 ->
// 156.1.  A W that stays in L2 from call to call only loses (82 MB: 24.8 ->
// 25.7 us; 41 MB 17.2 -> 18.0), and W below about this size does.  With no row
// masked they would be read for nothing, so all but kPrefetchAtOnce wait for a
// flag: 16 rows, none masked, of 2048, 32003 ids 6.5 us with all of them at once,
// 5.5 so, 5.2 with none at once, which costs the other calls (27.9 us) 0.5.
constexpr int kPrefetchBoxes = 16;
constexpr size_t kPrefetchMinBytes = 96u << 20;
// its ring: what is left of the 227 KB of a CTA next to its static shared
// memory (barriers and 2.5 KB of row statistics) and the 1 KB alignment
constexpr int kPairRingBytes = 222 * 1024;
constexpr size_t kPairSmemBytes = 1024 + kPairRingBytes;

// How many CTA pairs of `fn` the current device holds at once (0: none).
int head_pair_slots(const void* fn) {
  return sbd::cluster_slots(fn, kHeadThreads, kPairSmemBytes, 2);
}

// y = the sum over K ranges of the fp32 partials of sbd_linear, in bf16, each
// element in range order, with every range of an element requested at once.
// kVec: 4 outputs a thread, for T N a multiple of 4, where every range starts on
// 16 bytes, and from kReduceVec outputs on; fewer leave the threads too few: 1 to
// 64 rows of 1024 in 16 ranges, 4096 columns deep, 6.9-8.5 us with 4 outputs a
// thread, 6.4-7.8 with one; 128 rows of 4096 in 4 ranges 13.5 / 15.0.  (4 ranges
// requested at a time: those 1 to 64 rows 8.2-9.6 us.)
constexpr long long kReduceVec = 192 << 10;
template <int kRanges, bool kVec>
__global__ void __launch_bounds__(256)
linear_reduce_kernel(const float* __restrict__ part, long long tn, __nv_bfloat16* __restrict__ y) {
  grid_dependency_wait();
  grid_dependents_launch();
  const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * (kVec ? 4 : 1);
  if (i >= tn) return;
  if constexpr (kVec) {
    float4 v[kRanges];
#pragma unroll
    for (int ks = 0; ks < kRanges; ++ks)
      v[ks] = *reinterpret_cast<const float4*>(part + (size_t)ks * tn + i);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int ks = 0; ks < kRanges; ++ks) {
      acc.x += v[ks].x;
      acc.y += v[ks].y;
      acc.z += v[ks].z;
      acc.w += v[ks].w;
    }
    uint2 w;
    w.x = pack_bf16x2(acc.x, acc.y);
    w.y = pack_bf16x2(acc.z, acc.w);
    *reinterpret_cast<uint2*>(y + i) = w;
  } else {
    float v[kRanges];
#pragma unroll
    for (int ks = 0; ks < kRanges; ++ks) v[ks] = part[(size_t)ks * tn + i];
    float acc = 0.f;
#pragma unroll
    for (int ks = 0; ks < kRanges; ++ks) acc += v[ks];
    y[i] = __float2bfloat16_rn(acc);
  }
}

// The instance for a power of two of K ranges, 2 to 16.
template <bool kVec>
const void* linear_reduce_for(int ranges) {
  switch (ranges) {
    case 2: return (const void*)linear_reduce_kernel<2, kVec>;
    case 4: return (const void*)linear_reduce_kernel<4, kVec>;
    case 8: return (const void*)linear_reduce_kernel<8, kVec>;
    default: return (const void*)linear_reduce_kernel<16, kVec>;
  }
}

}  // namespace

namespace sbd {

HeadPlan head_plan(const sbd_head_desc& d) {
  HeadPlan p;
  p.B = d.batch;
  p.k = d.block_k;
  p.H = d.hidden;
  p.V = d.vocab;
  p.bf16 = d.dtype == SBD_DTYPE_BF16;
  const int bk = d.batch * d.block_k;
  p.rows_alloc = bk <= 16 ? 16 : ((bk + 15) / 16) * 16;
  const int n_tiles = (d.vocab + kBM - 1) / kBM;
  if (p.bf16) {
    const int slots = num_sms();
    p.n_ctas = n_tiles < slots ? n_tiles : slots;
  } else {
    p.n_ctas = n_tiles;
  }
  return p;
}

size_t head_workspace_bytes(const HeadPlan& p) { return head_ws_layout(p, nullptr).bytes; }

size_t head_workspace_floor(const sbd_head_desc& d) {
  if (d.batch < 0 || d.block_k < 1 || d.hidden < 1 || d.vocab < 1 ||
      (long long)d.batch * d.block_k > 512 ||
      (d.dtype != SBD_DTYPE_F32 && d.dtype != SBD_DTYPE_BF16))
    return 0;
  HeadPlan p;
  p.B = d.batch;
  p.k = d.block_k;
  p.H = d.hidden;
  p.V = d.vocab;
  p.bf16 = d.dtype == SBD_DTYPE_BF16;
  const int bk = d.batch * d.block_k;
  p.rows_alloc = bk <= 16 ? 16 : ((bk + 15) / 16) * 16;
  p.n_ctas = 1;
  return head_ws_layout(p, nullptr).bytes;
}

sbd_status head_launch(const HeadPlan& p, const void* hidden, const void* w,
                       const uint8_t* masked, const float* gumbel, float tau, float* entropy,
                       float* confidence, int32_t* token, void* ws, cudaStream_t st,
                       const PhiloxNoise* philox) {
  const int BK = p.B * p.k;
  if (BK == 0) return SBD_OK;
  if (tau == 0.f) philox = nullptr;                  // no noise
  HeadWs W = head_ws_layout(p, ws);
  sbd_status s;
  int* err = device_error_word();
  int n_parts = p.n_ctas;   // CTAs that write per-row partials
  if (p.bf16) {
    // CTA pairs from kPairMinRows allocated rows: as many as the device holds
    // at once, the pair tiles need and the workspace has partials for
    // (p.n_ctas), an even number when there may be two row groups.
    const bool few = BK <= kInPlaceRows;
    const void* fn_pair =
        philox ? (few               ? (const void*)head_pair_kernel<true, false, true>
                  : BK <= kFewRows  ? (const void*)head_pair_kernel<true, false, false, true>
                                    : (const void*)head_pair_kernel<true, false>)
               : (few               ? (const void*)head_pair_kernel<false, false, true>
                                    : (const void*)head_pair_kernel<false, false>);
    const int pair_tiles = (p.V + 2 * kBM - 1) / (2 * kBM);
    const int n_groups_max = p.rows_alloc > 2 * kPairRows ? 2 : 1;
    int n_pairs = 0;
    if (p.rows_alloc >= kPairMinRows && p.n_ctas >= 2) {
      n_pairs = head_pair_slots(fn_pair);
      if (n_pairs > pair_tiles * n_groups_max) n_pairs = pair_tiles * n_groups_max;
      if (n_pairs > p.n_ctas / 2) n_pairs = p.n_ctas / 2;
      if (n_groups_max == 2) n_pairs &= ~1;
    }
    const bool in_place = n_pairs > 0 && few;
    if (!in_place) {
      const uint8_t* hid = (const uint8_t*)hidden;
      int bk = BK, rb = p.H * 2;
      uint8_t* hc = W.hidden_c;
      int32_t* rm = W.row_map;
      int32_t* nr = W.n_rows;
      void* args[] = {(void*)&hid, (void*)&masked,  (void*)&bk,    (void*)&rb,
                      (void*)&hc,  (void*)&rm,      (void*)&nr,    (void*)&entropy,
                      (void*)&token, (void*)&confidence};
      s = launch_pdl((const void*)compact_rows_kernel, dim3(p.rows_alloc), dim3(256), 0, st, args,
                     "compact_rows_kernel launch");
      if (s != SBD_OK) return s;
    }
    CUtensorMap tw, th, th64, th128;
    {
      const uint64_t dims[2] = {(uint64_t)p.H, (uint64_t)p.V};
      const uint64_t strides[1] = {(uint64_t)p.H * 2};
      const uint32_t box[2] = {(uint32_t)kBK, (uint32_t)kBM};
      s = encode_tensor_map(&tw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)w, dims, strides,
                            box, CU_TENSOR_MAP_SWIZZLE_128B);
      if (s != SBD_OK) return s;
    }
    {
      void* rows = in_place ? (void*)hidden : (void*)W.hidden_c;
      const uint64_t dims[2] = {(uint64_t)p.H, (uint64_t)(in_place ? BK : p.rows_alloc)};
      const uint64_t strides[1] = {(uint64_t)p.H * 2};
      const uint32_t box[2] = {(uint32_t)kBK, 16u};
      s = encode_tensor_map(&th, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, rows, dims,
                            strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
      if (s != SBD_OK) return s;
      th64 = th;
      th128 = th;
      if (p.rows_alloc >= 64) {
        const uint32_t box64[2] = {(uint32_t)kBK, 64u};
        s = encode_tensor_map(&th64, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, rows, dims,
                              strides, box64, CU_TENSOR_MAP_SWIZZLE_128B);
        if (s != SBD_OK) return s;
      }
      if (p.rows_alloc >= 128) {
        const uint32_t box128[2] = {(uint32_t)kBK, 128u};
        s = encode_tensor_map(&th128, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, rows,
                              dims, strides, box128, CU_TENSOR_MAP_SWIZZLE_128B);
        if (s != SBD_OK) return s;
      }
    }
    HeadArgs a;
    a.gumbel = gumbel;
    a.seed_lo = philox ? (uint32_t)philox->seed : 0u;
    a.seed_hi = philox ? (uint32_t)(philox->seed >> 32) : 0u;
    a.off_lo = philox ? (uint32_t)philox->offset : 0u;
    a.off_hi = philox ? (uint32_t)(philox->offset >> 32) : 0u;
    a.row_map = W.row_map;
    a.n_rows = W.n_rows;
    a.masked = masked;
    a.n_flags = BK;
    a.prefetch = 0;
    if (in_place && (size_t)p.V * p.H * 2 >= kPrefetchMinBytes)
      a.prefetch = p.H / kBK < kPrefetchBoxes ? p.H / kBK : kPrefetchBoxes;
    a.row_map_out = W.row_map;
    a.n_rows_out = W.n_rows;
    a.entropy = entropy;
    a.token = token;
    a.confidence = confidence;
    a.part_msTb = W.part_msTb;
    a.part_idx = W.part_idx;
    a.err = err;
    a.V = p.V;
    a.H = p.H;
    a.rows_alloc = p.rows_alloc;
    a.n_tiles = (p.V + kBM - 1) / kBM;
    a.y = nullptr;
    a.linear_rows = 0;
    a.ksplit = 1;
    a.k_cluster = 0;
    a.w_rows = kBM;
    a.part_y = nullptr;
    a.h_big = p.rows_alloc >= 128 ? 128 : (p.rows_alloc >= 64 ? 64 : 16);
    a.tau = tau;
    const void* fn;
    size_t smem;
    if (n_pairs > 0) {
      fn = fn_pair;
      smem = kPairSmemBytes;
      a.ring_bytes = kPairRingBytes;
      a.n_tiles = pair_tiles;
      a.tmem_cols = 512;
      n_parts = 2 * n_pairs;
    } else {
      fn = philox ? (const void*)head_tc_kernel<true, false> : (const void*)head_tc_kernel<false, false>;
      smem = head_smem_bytes(p.rows_alloc);
      a.ring_bytes = head_ring_bytes(p.rows_alloc);
      // tensor memory for two accumulators of the allocated width (one of it
      // above 256 rows); the kernel picks the buffer count from the live rows
      const int n_acc_alloc = 2 * p.rows_alloc <= 512 ? 2 : 1;
      uint32_t cols = 32;
      while (cols < (uint32_t)(n_acc_alloc * p.rows_alloc)) cols <<= 1;
      a.tmem_cols = cols;
    }
    a.boxes = stage_boxes(p.H, 1);
    s = allow_smem(fn, smem, "cudaFuncSetAttribute(LM head kernel)");
    if (s != SBD_OK) return s;
    void* args[] = {(void*)&tw, (void*)&th, (void*)&th64, (void*)&th128, (void*)&a};
    s = launch_pdl(fn, dim3(n_parts), dim3(kHeadThreads), smem, st, args,
                   n_pairs > 0 ? "head_pair_kernel launch" : "head_tc_kernel launch",
                   n_pairs > 0 ? 2 : 1);
    if (s != SBD_OK) return s;
  } else {
    const float* hf = (const float*)hidden;
    const float* wf = (const float*)w;
    int bk = BK;
    int32_t* rm = W.row_map;
    int32_t* nr = W.n_rows;
    int V = p.V, H = p.H, ra = p.rows_alloc;
    float4* pm = W.part_msTb;
    int32_t* pi = W.part_idx;
    uint4 sk = make_uint4(0u, 0u, 0u, 0u);
    if (philox)
      sk = make_uint4((uint32_t)philox->seed, (uint32_t)(philox->seed >> 32),
                      (uint32_t)philox->offset, (uint32_t)(philox->offset >> 32));
    void* args[] = {(void*)&hf, (void*)&wf, (void*)&gumbel,  (void*)&masked, (void*)&bk,
                    (void*)&rm, (void*)&nr, (void*)&tau,     (void*)&V,      (void*)&H,
                    (void*)&ra, (void*)&pm, (void*)&pi,      (void*)&entropy, (void*)&token,
                    (void*)&confidence, (void*)&sk};
    const void* fn =
        philox ? (const void*)head_f32_kernel<true> : (const void*)head_f32_kernel<false>;
    s = allow_smem(fn, kF32SmemBytes, "cudaFuncSetAttribute(head_f32_kernel)");
    if (s != SBD_OK) return s;
    s = launch_pdl(fn, dim3(p.n_ctas), dim3(kF32HeadThreads), kF32SmemBytes, st, args, "head_f32_kernel launch");
    if (s != SBD_OK) return s;
  }
  {
    const float4* pm = W.part_msTb;
    const int32_t* pi = W.part_idx;
    int np = n_parts, ra = p.rows_alloc;
    const int32_t* rm = W.row_map;
    const int32_t* nr = W.n_rows;
    void* args[] = {(void*)&pm, (void*)&pi, (void*)&np,      (void*)&ra,   (void*)&rm,
                    (void*)&nr, (void*)&entropy, (void*)&token, (void*)&confidence};
    s = launch_pdl((const void*)head_combine_kernel, dim3((p.rows_alloc + 3) / 4), dim3(128), 0,
                   st, args, "head_combine_kernel launch");
    if (s != SBD_OK) return s;
  }
  return SBD_OK;
}

// y[T, N] = x[T, K] W[N, K]^T in bf16 with fp32 accumulation: the LM-head
// kernel's main loop (W streamed once through the ring, x's rows from L2)
// with a storing epilogue.
// The largest K split sbd_linear may use: powers of two up to 16, each K
// range at least 4 column blocks long, at most 512 (tile, range) units and
// at most 64 MB of fp32 partials.  A function of the shape only, so that
// the workspace size does not depend on the device.
static int linear_max_split(int T, int K, int N) {
  const int kb64 = K / kBK, n_tiles = (N + kBM - 1) / kBM;
  int ks = 1;
  while (ks < 16 && kb64 % (2 * ks) == 0 && kb64 / (2 * ks) >= 4 &&
         (long long)n_tiles * 2 * ks <= 512 &&
         (long long)2 * ks * T * N * (long long)sizeof(float) <= (64ll << 20))
    ks *= 2;
  return ks;
}

int linear_ksplit(int T, int K, int N) {
  // A time model per SM: a tile streams its 128 x K weights (~45 GB/s per
  // SM at the HBM peak) or runs its 2 x 128 x n x K flops (~14.8 TFLOP/s
  // per SM), whichever is longer; a unit of a split also writes its
  // T x 128 fp32 partials, and the sum over ranges reads them all back in
  // a second launch.  The split with the shortest modelled time wins.
  const int max_ks = linear_max_split(T, K, N);
  const int sms = num_sms();
  const int n_tiles = (N + kBM - 1) / kBM;
  const double n_eff = T <= 16 ? 16.0 : (double)((T + 15) / 16 * 16);
  const double t_mem = 128.0 * K * 2 / 45e3, t_mma = 2.0 * 128 * n_eff * K / 14.8e6;  // us
  const double t_tile = t_mem > t_mma ? t_mem : t_mma;
  const double t_part = (double)T * 128 * 4 / 45e3;
  int best = 1;
  double best_cost = (double)((n_tiles + sms - 1) / sms) * t_tile;
  for (int ks = 2; ks <= max_ks; ks *= 2) {
    const double waves = (double)((n_tiles * ks + sms - 1) / sms);
    const double cost = waves * (t_tile / ks + t_part) + (double)ks * T * N * 4 / 6e6 + 2.0;
    if (cost < best_cost) {
      best_cost = cost;
      best = ks;
    }
  }
  return best;
}

// W rows per CTA and unit, and K ranges, of the CTA-pair linear: the pair of
// shortest modelled time.  A 64-column block of a unit takes as long as its
// rows' fill of shared memory (107 GB/s an SM, measured in the main loop at
// 512 rows) or its four 2-SM MMAs (44 ns up to N = 128, 65 at N = 256), and no
// less than 0.235 us (measured at 32 and 64 W rows); units go to the pairs of
// their row group in rounds.  Fewer W rows a unit fill a round better (512 x
// 6144, 38 pairs a group: 24 units of 256 ids, 32 of 192); K ranges shorten the
// units but write fp32 partials that a second kernel reads back.  At most
// linear_max_split ranges (what the workspace holds).  Against 128 W rows
// throughout (an 8B layer's four GEMMs): 256 rows 126.0 -> 120.4 us, 512 rows
// 165.3 -> 162.5 in bursts.
struct PairSplit {
  int w_rows, ksplit;
};
static PairSplit pair_linear_split(int T, int K, int N, int n_pairs) {
  const int max_ks = linear_max_split(T, K, N);
  const int n_groups = T > 2 * kPairRows ? 2 : 1;
  const int per_group = n_pairs / n_groups > 0 ? n_pairs / n_groups : 1;
  const int live = T < kPairRows ? T : kPairRows;
  PairSplit best = {kBM, 1};
  double best_cost = 1e30;
  for (int wr = kBM; wr >= 32; wr -= 16) {
    const int tiles = (N + 2 * wr - 1) / (2 * wr);
    const double fill = (live + wr) * 128.0 / 107e3;   // us
    const double mma = 4 * (wr <= 64 ? 0.0441 : 0.0441 + (2 * wr - 128) / 128.0 * 0.0213);
    const double t_blk = fill > mma ? (fill > 0.235 ? fill : 0.235) : (mma > 0.235 ? mma : 0.235);
    for (int ks = 1; ks <= max_ks; ks *= 2) {
      const int rounds = (tiles * ks + per_group - 1) / per_group;
      double cost = rounds * (t_blk * (K / kBK / ks) + 0.5) + wr * (ks > 1 ? 0.02 : 0.016);
      if (ks > 1) cost += (double)ks * T * N * 4 / 12e6 + 1.5;
      if (cost < best_cost) {
        best_cost = cost;
        best = {wr, ks};
      }
    }
  }
  return best;
}

// K ranges of the single-CTA linear kernel's tiles as clusters, all running at
// once (1: through the workspace): as many as the SMs hold, each at least 4
// column blocks, of even length.  The ranges then add up through distributed
// shared memory, with no fp32 partials in HBM and no second kernel: 4096 -> 4096
// columns at 128 rows 13.5 -> 12.6 us, at 160 rows 16.3 -> 14.6, 4096 -> 6144 17.9
// -> 17.2, 22.3 -> 20.9; 1024 -> 1024 at 16 rows 6.1 -> 5.7.  Where clusters cannot
// be as many CTAs as the split through the workspace (8 a tile at most, and what
// fits in the GPU's parts) that one is taken: 2048 -> 2048 at 1 row 7.4 us in
// clusters of 7, 6.3 in 8 ranges; 8192 -> 2048 at 64 rows 13.1 / 11.8.
static int linear_cluster_ranges(const void* fn, size_t smem, int T, int K, int n_tiles, int ksplit) {
  if (T > kPairVocabLanesMax) return 1;   // T x 128 partials fit the ring
  const int pairs = (K / kBK) % 2 == 0 ? 2 : 1;         // boxes of a stage: two, where even
  // (Through the workspace the units go to the SMs in rounds, so many at a time;
  // three quarters of that in clusters, one launch with the next one's W on its way,
  // are as good: the GEMMs of a layer of 3072 and 8192 columns, 48 rows 57.4 -> 55.4 us,
  // of an 8B layer, 16 rows 86.2 -> 84.8, though 4096 -> 6144 by itself 12.8 -> 13.3 at
  // 1 row.  With a single round not: 8192 -> 2048 at 1 row, 128 CTAs 9.5, 112 11.3.)
  const int sms = num_sms(), units = n_tiles * ksplit, rounds = (units + sms - 1) / sms;
  const int in_ws = rounds == 1 ? units : 3 * units / (4 * rounds);
  for (int ks = kMaxRanges; ks > 1 && n_tiles * ks >= in_ws; --ks)
    if (n_tiles * ks <= sms && K / kBK >= 4 * ks && even_ranges(K / kBK / pairs, ks) &&
        cluster_slots(fn, kHeadThreads, smem, ks) >= n_tiles)
      return ks;
  return 1;
}

size_t linear_workspace_bytes(int T, int K, int N) {
  const int ks = linear_max_split(T, K, N);
  return ks > 1 ? (size_t)ks * T * N * sizeof(float) : 0;
}

sbd_status linear_launch(int T, int K, int N, const void* x, const void* w, void* y, void* ws,
                         cudaStream_t st) {
  if (T == 0 || N == 0) return SBD_OK;
  const int rows_alloc = T <= 16 ? 16 : ((T + 15) / 16) * 16;
  CUtensorMap tw, tx, tx64, tx128;
  sbd_status s;
  {
    const uint64_t dims[2] = {(uint64_t)K, (uint64_t)N};
    const uint64_t strides[1] = {(uint64_t)K * 2};
    const uint32_t box[2] = {(uint32_t)kBK, (uint32_t)kBM};
    s = encode_tensor_map(&tw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)w, dims, strides, box,
                          CU_TENSOR_MAP_SWIZZLE_128B);
    if (s != SBD_OK) return s;
  }
  {
    // rows of x past T (up to the MMA's multiple of 16) are read as zeros
    const uint64_t dims[2] = {(uint64_t)K, (uint64_t)T};
    const uint64_t strides[1] = {(uint64_t)K * 2};
    const uint32_t box[2] = {(uint32_t)kBK, 16u};
    s = encode_tensor_map(&tx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)x, dims, strides, box,
                          CU_TENSOR_MAP_SWIZZLE_128B);
    if (s != SBD_OK) return s;
    tx64 = tx;
    tx128 = tx;
    if (T >= 64) {
      const uint32_t box64[2] = {(uint32_t)kBK, 64u};
      s = encode_tensor_map(&tx64, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)x, dims, strides,
                            box64, CU_TENSOR_MAP_SWIZZLE_128B);
      if (s != SBD_OK) return s;
    }
    if (T >= 128) {
      const uint32_t box128[2] = {(uint32_t)kBK, 128u};
      s = encode_tensor_map(&tx128, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)x, dims, strides,
                            box128, CU_TENSOR_MAP_SWIZZLE_128B);
      if (s != SBD_OK) return s;
    }
  }
  HeadArgs a{};
  a.err = device_error_word();
  a.V = N;
  a.H = K;
  a.rows_alloc = rows_alloc;
  a.n_tiles = (N + kBM - 1) / kBM;
  a.k_cluster = 0;
  a.w_rows = kBM;
  a.h_big = T >= 128 ? 128 : (T >= 64 ? 64 : 16);
  a.tau = 0.f;
  a.y = (__nv_bfloat16*)y;
  a.linear_rows = T;
  a.part_y = (float*)ws;
  // Above the pair kernel's vocabulary-lane limit: CTA pairs in the rows
  // layout, as many as the device holds at once and the units need (an
  // even number with two row groups), with their own choice of K ranges.
  int ksplit = linear_ksplit(T, K, N);
  const void* fn = nullptr;
  int n_ctas = 0, cluster = 1;
  size_t smem = 0;
  if (T > kPairVocabLanesMax) {
    const void* fn_pair = (const void*)head_pair_kernel<false, true>;
    const int n_groups = T > 2 * kPairRows ? 2 : 1;
    int n_pairs = head_pair_slots(fn_pair);
    if (n_groups == 2) n_pairs &= ~1;
    if (n_pairs > 0) {
      const PairSplit sp = pair_linear_split(T, K, N, n_pairs);
      const int ks = sp.ksplit, pair_tiles = (N + 2 * sp.w_rows - 1) / (2 * sp.w_rows);
      if (n_pairs > pair_tiles * n_groups * ks) n_pairs = pair_tiles * n_groups * ks;
      if (n_groups == 2) n_pairs &= ~1;
      if (n_pairs > 0) {
        ksplit = ks;
        a.w_rows = sp.w_rows;
        if (sp.w_rows != kBM) {
          const uint32_t box_w[2] = {(uint32_t)kBK, (uint32_t)sp.w_rows};
          const uint64_t dims[2] = {(uint64_t)K, (uint64_t)N};
          const uint64_t strides[1] = {(uint64_t)K * 2};
          s = encode_tensor_map(&tw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)w, dims, strides,
                                box_w, CU_TENSOR_MAP_SWIZZLE_128B);
          if (s != SBD_OK) return s;
        }
        fn = fn_pair;
        n_ctas = 2 * n_pairs;
        cluster = 2;
        smem = kPairSmemBytes;
        a.n_tiles = pair_tiles;
        a.ring_bytes = kPairRingBytes;
        a.tmem_cols = 512;
      }
    }
  }
  if (!fn) {
    fn = (const void*)head_tc_kernel<false, true>;
    smem = head_smem_bytes(rows_alloc);
    a.ring_bytes = head_ring_bytes(rows_alloc);
    const int n_acc_alloc = 2 * rows_alloc <= 512 ? 2 : 1;
    uint32_t cols = 32;
    while (cols < (uint32_t)(n_acc_alloc * rows_alloc)) cols <<= 1;
    a.tmem_cols = cols;
    const int slots = num_sms();
    const int in_cluster = linear_cluster_ranges(fn, smem, T, K, a.n_tiles, ksplit);
    if (in_cluster > 1) {
      ksplit = in_cluster;
      a.k_cluster = 1;
      cluster = ksplit;
    }
    const int units = a.n_tiles * ksplit;
    n_ctas = a.k_cluster || units < slots ? units : slots;
  }
  a.ksplit = ksplit;
  a.boxes = stage_boxes(K, ksplit);
  s = allow_smem(fn, smem, "cudaFuncSetAttribute(linear kernel)");
  if (s != SBD_OK) return s;
  void* args[] = {(void*)&tw, (void*)&tx, (void*)&tx64, (void*)&tx128, (void*)&a};
  s = launch_pdl(fn, dim3(n_ctas), dim3(kHeadThreads), smem, st, args,
                 T > kPairVocabLanesMax ? "head_pair_kernel (linear) launch" : "head_tc_kernel (linear) launch",
                 cluster);
  if (s != SBD_OK || ksplit == 1 || a.k_cluster) return s;
  const float* part = (const float*)ws;
  long long tn = (long long)T * N;
  __nv_bfloat16* yb = (__nv_bfloat16*)y;
  void* rargs[] = {(void*)&part, (void*)&tn, (void*)&yb};
  const bool vec = tn % 4 == 0 && tn >= kReduceVec;
  const long long threads = vec ? tn / 4 : tn;
  return launch_pdl(vec ? linear_reduce_for<true>(ksplit) : linear_reduce_for<false>(ksplit),
                    dim3((unsigned)((threads + 255) / 256)), dim3(256), 0, st, rargs,
                    "linear_reduce_kernel launch");
}

}  // namespace sbd
