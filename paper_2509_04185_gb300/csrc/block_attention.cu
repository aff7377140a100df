// Block attention of one SBD forward (arXiv 2509.04185, Eq. 5; inference
// mask of Fig. 3): the k block queries of a sequence attend to its exact KV
// cache (all of it lies in their past) and bidirectionally to the k block
// keys.  This file holds the plan (KV splits per (sequence, KV head), the
// in-cluster merge or the workspace), the launch, the split merge kernel
// for plans whose splits do not form a cluster, and the fp32 variant; the
// bf16 kernels are the tcgen05 ones of block_attention_tc.cu:
//
//   * one CTA per (KV split, KV head, sequence); the G = Hq/Hkv query heads
//     that share a KV head are packed with the k block rows into one
//     M = G*k row tile (row r = i*G + g), so each K/V byte is read once;
//   * with more than one split, each CTA's normalised partial output and
//     log-sum-exp are merged inside its thread-block cluster, or written to
//     the workspace and merged by attn_combine_kernel.
//
// First iteration of a block after the previous one (Algorithm 3, "first
// iteration and t >= k"): the leading n_causal block rows are the previous
// block's tokens, causal among themselves, and their keys/values are written
// into the cache at L_b .. L_b + n_causal - 1 by the warp that brings the
// block tile in.
//
// The fp32 variant (attn_f32_kernel) runs on fp32 FMAs throughout, split over
// key ranges with the same in-cluster merge.
#include <math.h>

#include "sbd_internal.cuh"

namespace {

using namespace sbd_dev;

constexpr int kTileKeys = 64;
// Largest batch for which the CTAs of a multi-wave launch take the
// sequences longest first.
constexpr int kOrderMaxB = 128;
constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// Merge of the split partials: O = sum_s 2^(lse_s - lse) O_s.  One warp per
// (packed row, KV head, sequence), kCombineRows rows per CTA: lane s holds
// the log-sum-exp of split s, and each lane owns D / 32 consecutive output
// columns.  The kernel is latency-bound: for each group of 32 splits a lane
// requests the log-sum-exp and its columns of all of them before it uses
// any, so that one memory round trip covers the group; groups merge online.
// (One 128-thread CTA per row instead took 12.6 us for 2048 CTAs at 4
// splits, its time growing with the CTA count.)
constexpr int kCombineRows = 4;

template <int D, typename OutT>
__global__ void __launch_bounds__(32 * kCombineRows)
attn_combine_kernel(const float* __restrict__ part_o, const float* __restrict__ part_lse,
                    OutT* __restrict__ out, int k, int Hq, int Hkv, int G, int M, int splits) {
  constexpr int kPer = D / 32;                 // columns per lane: 2 or 4
  grid_dependency_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.x * kCombineRows + warp, hkv = blockIdx.y, b = blockIdx.z;
  if (r >= M) return;
  const size_t pair = (size_t)b * Hkv + hkv;
  const float* lse = part_lse + pair * splits * M + r;
  const float* po = part_o + (pair * splits * M + r) * D + kPer * lane;
  const size_t po_stride = (size_t)M * D;
  float mx = -INFINITY, sum = 0.f, acc[kPer];
#pragma unroll
  for (int c = 0; c < kPer; ++c) acc[c] = 0.f;
  for (int s0 = 0; s0 < splits; s0 += 32) {
    const int n = min(32, splits - s0);
    const float l_lane = lane < n ? lse[(size_t)(s0 + lane) * M] : -INFINITY;
    float v[32][kPer];
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      if (e < n) {
        const float* src = po + (size_t)(s0 + e) * po_stride;
        if constexpr (kPer == 4) {
          const float4 x = *reinterpret_cast<const float4*>(src);
          v[e][0] = x.x; v[e][1] = x.y; v[e][2] = x.z; v[e][3] = x.w;
        } else {
          const float2 x = *reinterpret_cast<const float2*>(src);
          v[e][0] = x.x; v[e][1] = x.y;
        }
      } else {
#pragma unroll
        for (int c = 0; c < kPer; ++c) v[e][c] = 0.f;
      }
    }
    const float gm = warp_max(l_lane);
    if (gm == -INFINITY) continue;               // every split of the group is empty
    if (gm > mx) {
      const float c = exp2f(mx - gm);            // 0 while mx = -inf
      sum *= c;
#pragma unroll
      for (int e = 0; e < kPer; ++e) acc[e] *= c;
      mx = gm;
    }
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      const float wt = exp2f(__shfl_sync(0xffffffffu, l_lane, e) - mx);   // 0 past n
      sum += wt;
      if (wt > 0.f) {
#pragma unroll
        for (int c = 0; c < kPer; ++c) acc[c] = fmaf(wt, v[e][c], acc[c]);
      }
    }
  }
  const float inv = sum > 0.f ? 1.f / sum : 0.f;
  const size_t o = (((size_t)b * k + r / G) * Hq + hkv * G + r % G) * D + kPer * lane;
  if constexpr (sizeof(OutT) == 2) {
    if constexpr (kPer == 4) {
      uint2 w;
      w.x = pack_bf16(acc[0] * inv, acc[1] * inv);
      w.y = pack_bf16(acc[2] * inv, acc[3] * inv);
      *reinterpret_cast<uint2*>(out + o) = w;
    } else {
      *reinterpret_cast<uint32_t*>(out + o) = pack_bf16(acc[0] * inv, acc[1] * inv);
    }
  } else {
#pragma unroll
    for (int c = 0; c < kPer; ++c) out[o + c] = acc[c] * inv;
  }
}

// ------------------------------------------------------------ fp32 variant
// Split-KV attention on fp32 FMAs.  One CTA per (key range, KV head,
// sequence, chunk of W RW packed rows r = i*G + g): keys pass through shared
// memory in tiles of 64, each K/V element read from global memory once per
// row chunk.  A warp owns RW rows in both products, so the softmax and P stay
// inside the warp:
//   S   lane = keys (lane, lane + 32) of the tile; Q rows are broadcast
//       reads;
//   P   through shared memory within the warp;
//   O   lane = D / 32 consecutive dimensions; P values are broadcast reads.
// The key ranges of a (sequence, KV head, chunk) are the CTAs of one
// thread-block cluster and merge through distributed shared memory, so no
// workspace is needed.
// Bound: the FMAs of a full tile are 2 us of an SM (32 rows x 64 keys x 128
// dimensions, twice); a tile measured 5.2 us with one CTA on the SM, the rest
// being latencies between the phases, which a second CTA covers in part, and
// reads of shared memory (S: 12 cycles of its port for 8 of FMAs; PV: 20 for
// 16).  With 4 warps of 8 rows in place of 8 of 4: 6 % slower at the shape below.
// The form before (one CTA per query row and head, each walking all keys,
// uncoalesced) took 717 us at B = 2, k = 8, 32/8 heads of 128, 511-2048
// cached keys, and 37 us at 4/2 heads of 64, k = 4, 128 keys (the smallest
// configuration); this one takes 27-29 us by the lengths drawn, and 4.7 (the FMAs
// of the first are 4.2 us of the whole chip, its bytes 3.1 us of HBM).
constexpr int kF32Keys = 64;                 // keys per tile
constexpr int kF32Granule = 16;              // key ranges are multiples of this

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A float at this CTA's shared location `p`, read in CTA `rank` of the cluster.
__device__ __forceinline__ float ld_rank(const float* p, int rank) {
  uint32_t a;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_rank2(const float* p, int rank) {
  uint32_t a;
  float2 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}

struct F32Args {
  const float *q, *kc, *vc;
  const int32_t* lens;
  const float *kb, *vb;
  float* out;
  int* err;
  float *kc_app, *vc_app;      // writable caches for the causal rows, or NULL
  int k, Hq, Hkv, G, M, Lmax, n_causal, splits, chunks;
  float scale_log2;
};

template <int D>
__host__ __device__ constexpr int f32_k_stride() { return D + 4; }   // lanes' rows in distinct banks

template <int D, int RW, int W>
constexpr size_t f32_smem_bytes() {
  return sizeof(float) * ((size_t)W * RW * D                            // Q
                          + (size_t)kF32Keys * (f32_k_stride<D>() + D)  // K, V tile
                          + (size_t)W * RW * kF32Keys                   // P
                          + 2 * W * RW);                                // m, l of the merge
}

// Registers: shared memory holds two CTAs of 256 threads an SM, but left to
// itself the compiler cuts its loads short to fit three (80 registers): 9 rows
// x 4 heads of 64, batch 3, 1000 keys 18.8 us with 96 registers, 20.9 with 80,
// 19.8 with 128; 2 rows x 3 heads of 128, batch 1, 2000 keys 9.6 with 128, 10.4
// with 64.
template <int D, int RW, int W>
__global__ void __maxnreg__(D == 64 && RW == 4 ? 96 : 128)
attn_f32_kernel(const F32Args a) {
  constexpr int kF32Warps = W, kF32Threads = 32 * W;
  constexpr int kRowsCta = kF32Warps * RW;
  constexpr int kKS = f32_k_stride<D>();
  constexpr int kPer = D / 32;                 // output dimensions per lane
  constexpr int kC4 = D / 4;                   // 16-byte chunks of a row
  extern __shared__ __align__(16) float sm[];
  float* q_s = sm;                             // [kRowsCta][D]
  float* k_s = q_s + kRowsCta * D;             // [kF32Keys][kKS]
  float* v_s = k_s + kF32Keys * kKS;           // [kF32Keys][D]
  float* p_s = v_s + kF32Keys * D;             // [kRowsCta][kF32Keys]
  float* st_s = p_s + kRowsCta * kF32Keys;     // m, then l: [kRowsCta] each
  float* o_s = k_s;                            // merge: [kRowsCta][D], over the dead K tile
  static_assert(kRowsCta * D <= kF32Keys * kKS, "the partial rows fit the K tile");

  grid_dependency_wait();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int split = blockIdx.x, hkv = blockIdx.y / a.chunks, chunk = blockIdx.y % a.chunks;
  const int b = blockIdx.z;
  int len = a.lens[b];
  if (len < 0 || len > a.Lmax) {
    if (tid == 0) record_error(a.err, SBD_DEVERR_CACHE_LEN);
    len = len < 0 ? 0 : a.Lmax;
  }
  const int total = len + a.k;
  const int range = ((total + a.splits - 1) / a.splits + kF32Granule - 1) / kF32Granule * kF32Granule;
  const int u_begin = min(total, split * range), u_end = min(total, u_begin + range);

  // Cache and block rows are both Hkv * D floats apart; a thread always
  // copies the same 16-byte column of a row.
  const int row_floats = a.Hkv * D;
  const int c_ld = 4 * (tid % kC4), j_ld = tid / kC4;
  const size_t cache_off = ((size_t)b * a.Lmax * a.Hkv + hkv) * D + c_ld;
  const size_t blk_off = ((size_t)b * a.k * a.Hkv + hkv) * D + c_ld;
  auto load_tile = [&](float* dst, int stride, const float* cache, const float* blk, int t0) {
    // rows up to the next multiple of 4 keys are zeros (PV takes 4 at a time)
    const int n4 = (min(kF32Keys, u_end - t0) + 3) & ~3;
#pragma unroll 4
    for (int j = j_ld; j < n4; j += kF32Threads / kC4) {
      const int u = t0 + j;
      const bool valid = u < u_end;
      const float* src = u < len ? cache + cache_off + (size_t)u * row_floats
                                 : blk + blk_off + (size_t)(valid ? u - len : 0) * row_floats;
      cp_async16(dst + j * stride + c_ld, src, valid);
    }
    cp_async_commit();
  };
  if (u_begin < u_end) load_tile(k_s, kKS, a.kc, a.kb, u_begin);

  // Q rows of the chunk (zeros past M)
  for (int e = tid; e < kRowsCta * kC4; e += kF32Threads) {
    const int rl = e / kC4, c = e % kC4, r = chunk * kRowsCta + rl;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < a.M)
      v = *reinterpret_cast<const float4*>(
          a.q + (((size_t)b * a.k + r / a.G) * a.Hq + hkv * a.G + r % a.G) * D + 4 * c);
    *reinterpret_cast<float4*>(q_s + rl * D + 4 * c) = v;
  }
  // The first CTA of each (sequence, KV head) writes the causal rows' keys
  // and values into the cache; cache positions < len alone are read.
  if (a.kc_app && split == 0 && chunk == 0) {
    if (len + a.n_causal <= a.Lmax) {
      for (int e = tid; e < a.n_causal * kC4; e += kF32Threads) {
        const int i = e / kC4, c = e % kC4;
        const size_t dst = (((size_t)b * a.Lmax + len + i) * a.Hkv + hkv) * D + 4 * c;
        const size_t src = (((size_t)b * a.k + i) * a.Hkv + hkv) * D + 4 * c;
        *reinterpret_cast<float4*>(a.kc_app + dst) = *reinterpret_cast<const float4*>(a.kb + src);
        *reinterpret_cast<float4*>(a.vc_app + dst) = *reinterpret_cast<const float4*>(a.vb + src);
      }
    } else if (tid == 0) {
      record_error(a.err, SBD_DEVERR_CACHE_LEN);
    }
  }

  // this warp's rows: local rows RW*warp .. + RW - 1; keys u < vis[r] are seen
  int vis[RW], vis_min = u_end;
#pragma unroll
  for (int r = 0; r < RW; ++r) {
    const int i = (chunk * kRowsCta + RW * warp + r) / a.G;
    vis[r] = min(u_end, len + (i < a.n_causal ? i + 1 : a.k));
    vis_min = min(vis_min, vis[r]);
  }
  float m[RW], l[RW];                          // l: this lane's share of the row sum
  float o[RW][kPer];
#pragma unroll
  for (int r = 0; r < RW; ++r) {
    m[r] = -INFINITY;
    l[r] = 0.f;
#pragma unroll
    for (int c = 0; c < kPer; ++c) o[r][c] = 0.f;
  }
  const float* qw = q_s + RW * warp * D;
  float* pw = p_s + RW * warp * kF32Keys;

  for (int t0 = u_begin; t0 < u_end; t0 += kF32Keys) {
    const int n = min(kF32Keys, u_end - t0);
    load_tile(v_s, D, a.vc, a.vb, t0);
    cp_async_wait<1>();                        // the K tile
    __syncthreads();
    // ---- S: keys lane and lane + 32 of the tile
    const bool two = n > 32;
    float s[RW][2];
    {
      float acc[RW][2];
#pragma unroll
      for (int r = 0; r < RW; ++r) acc[r][0] = acc[r][1] = 0.f;
      const float* k0 = k_s + lane * kKS;
      const float* k1 = k0 + 32 * kKS;
      if (two) {
#pragma unroll 4
        for (int c = 0; c < kC4; ++c) {
          const float4 x0 = *reinterpret_cast<const float4*>(k0 + 4 * c);
          const float4 x1 = *reinterpret_cast<const float4*>(k1 + 4 * c);
#pragma unroll
          for (int r = 0; r < RW; ++r) {
            const float4 qv = *reinterpret_cast<const float4*>(qw + r * D + 4 * c);
            acc[r][0] = dot4(qv, x0, acc[r][0]);
            acc[r][1] = dot4(qv, x1, acc[r][1]);
          }
        }
      } else {
#pragma unroll 4
        for (int c = 0; c < kC4; ++c) {
          const float4 x0 = *reinterpret_cast<const float4*>(k0 + 4 * c);
#pragma unroll
          for (int r = 0; r < RW; ++r)
            acc[r][0] = dot4(*reinterpret_cast<const float4*>(qw + r * D + 4 * c), x0, acc[r][0]);
        }
      }
      // keys past the row's last visible one (their tile rows may hold
      // anything) do not count
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        s[r][0] = t0 + lane < vis[r] ? acc[r][0] * a.scale_log2 : -INFINITY;
        s[r][1] = two && t0 + lane + 32 < vis[r] ? acc[r][1] * a.scale_log2 : -INFINITY;
      }
    }
    // ---- softmax of the tile
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const float mn = fmaxf(m[r], warp_max(fmaxf(s[r][0], s[r][1])));
      const float alpha = m[r] == -INFINITY ? 0.f : exp2f(m[r] - mn);
      const float p0 = s[r][0] == -INFINITY ? 0.f : exp2f(s[r][0] - mn);
      const float p1 = s[r][1] == -INFINITY ? 0.f : exp2f(s[r][1] - mn);
      m[r] = mn;
      l[r] = fmaf(l[r], alpha, p0 + p1);
#pragma unroll
      for (int c = 0; c < kPer; ++c) o[r][c] *= alpha;
      pw[r * kF32Keys + lane] = p0;
      pw[r * kF32Keys + lane + 32] = p1;
    }
    cp_async_wait<0>();                        // the V tile
    __syncthreads();                           // every warp is done with the K tile, too
    if (t0 + kF32Keys < u_end) load_tile(k_s, kKS, a.kc, a.kb, t0 + kF32Keys);
    // ---- O += P V, 4 keys at a time, as far as every row of the warp sees them
    const int n_all = t0 + n <= vis_min ? n : max(0, vis_min - t0) & ~3;
#pragma unroll 2
    for (int j = 0; j < n_all; j += 4) {
      float v[4][kPer];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if constexpr (kPer == 4) {
          const float4 x = *reinterpret_cast<const float4*>(v_s + (j + e) * D + 4 * lane);
          v[e][0] = x.x, v[e][1] = x.y, v[e][2] = x.z, v[e][3] = x.w;
        } else {
          const float2 x = *reinterpret_cast<const float2*>(v_s + (j + e) * D + 2 * lane);
          v[e][0] = x.x, v[e][1] = x.y;
        }
      }
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const float4 p = *reinterpret_cast<const float4*>(pw + r * kF32Keys + j);
#pragma unroll
        for (int c = 0; c < kPer; ++c) {
          o[r][c] = fmaf(p.x, v[0][c], o[r][c]);
          o[r][c] = fmaf(p.y, v[1][c], o[r][c]);
          o[r][c] = fmaf(p.z, v[2][c], o[r][c]);
          o[r][c] = fmaf(p.w, v[3][c], o[r][c]);
        }
      }
    }
    // The rest, block keys that some causal row must not see: their values are
    // left out there, not multiplied by 0 (they may be infinite or NaN).
#pragma unroll 1
    for (int j = n_all; j < n; ++j) {
      float v[kPer];
#pragma unroll
      for (int c = 0; c < kPer; ++c) v[c] = v_s[j * D + kPer * lane + c];
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        if (t0 + j >= vis[r]) continue;
        const float p = pw[r * kF32Keys + j];
#pragma unroll
        for (int c = 0; c < kPer; ++c) o[r][c] = fmaf(p, v[c], o[r][c]);
      }
    }
    __syncthreads();                           // the V tile is consumed
  }
  grid_dependents_launch();

  auto store_row = [&](int rl, const float (&x)[kPer], float sum) {
    const int r = chunk * kRowsCta + rl;
    if (r >= a.M) return;
    float* dst = a.out + (((size_t)b * a.k + r / a.G) * a.Hq + hkv * a.G + r % a.G) * D + kPer * lane;
#pragma unroll
    for (int c = 0; c < kPer; c += 2)
      *reinterpret_cast<float2*>(dst + c) = make_float2(x[c] / sum, x[c + 1] / sum);
  };
  if (a.splits == 1) {
#pragma unroll
    for (int r = 0; r < RW; ++r) store_row(RW * warp + r, o[r], warp_sum(l[r]));
    return;
  }
  // ---- merge over the cluster: every CTA leaves its rows' maximum, sum and
  // unnormalised O in shared memory; CTA `split` merges rows split,
  // split + splits, ...  The second barrier keeps shared memory alive until
  // every CTA has read it.
  __syncthreads();
#pragma unroll
  for (int r = 0; r < RW; ++r) {
    const int rl = RW * warp + r;
    const float lr = warp_sum(l[r]);
#pragma unroll
    for (int c = 0; c < kPer; c += 2)
      *reinterpret_cast<float2*>(o_s + rl * D + kPer * lane + c) = make_float2(o[r][c], o[r][c + 1]);
    if (lane == 0) {
      st_s[rl] = m[r];
      st_s[kRowsCta + rl] = lr;
    }
  }
  cluster_sync_all();
  for (int rl = split + a.splits * warp; rl < kRowsCta && chunk * kRowsCta + rl < a.M;
       rl += a.splits * kF32Warps) {
    const float ms = lane < a.splits ? ld_rank(st_s + rl, lane) : -INFINITY;
    const float ls = lane < a.splits ? ld_rank(st_s + kRowsCta + rl, lane) : 0.f;
    const float mx = warp_max(ms);
    const float w = mx == -INFINITY ? (lane < a.splits ? 1.f : 0.f) : exp2f(ms - mx);
    const float lsum = warp_sum(w * ls);
    float acc[kPer];
#pragma unroll
    for (int c = 0; c < kPer; ++c) acc[c] = 0.f;
#pragma unroll 4
    for (int e = 0; e < a.splits; ++e) {
      const float we = __shfl_sync(0xffffffffu, w, e);
#pragma unroll
      for (int c = 0; c < kPer; c += 2) {
        const float2 x = ld_rank2(o_s + rl * D + kPer * lane + c, e);
        acc[c] = fmaf(we, x.x, acc[c]);
        acc[c + 1] = fmaf(we, x.y, acc[c + 1]);
      }
    }
    store_row(rl, acc, lsum);
  }
  cluster_sync_all();
}

// The instance for M packed rows: few rows per warp at small M (a small block
// keeps every warp busy), else chunks of 32 rows on 8 warps.
struct F32Kernel {
  const void* fn;
  size_t smem;
  int rows;          // packed rows per CTA
  int threads;
};
F32Kernel f32_kernel_for(int D, int M) {
  if (D == 128) {
    if (M <= 8) return {(const void*)attn_f32_kernel<128, 2, 4>, f32_smem_bytes<128, 2, 4>(), 8, 128};
    if (M <= 16) return {(const void*)attn_f32_kernel<128, 4, 4>, f32_smem_bytes<128, 4, 4>(), 16, 128};
    return {(const void*)attn_f32_kernel<128, 4, 8>, f32_smem_bytes<128, 4, 8>(), 32, 256};
  }
  if (M <= 8) return {(const void*)attn_f32_kernel<64, 2, 4>, f32_smem_bytes<64, 2, 4>(), 8, 128};
  if (M <= 16) return {(const void*)attn_f32_kernel<64, 4, 4>, f32_smem_bytes<64, 4, 4>(), 16, 128};
  return {(const void*)attn_f32_kernel<64, 4, 8>, f32_smem_bytes<64, 4, 8>(), 32, 256};
}

}  // namespace

namespace sbd {

// KV splits per (sequence, KV head): one wave of CTAs, each as long as
// possible.  A CTA pays a fixed start (tensor memory, barriers, Q, the first
// loads' latency) and drain; measured on the long-cache workloads, filling
// further waves with shorter CTAs loses more than the idle SMs of one wave.
static int choose_splits(int pairs, int n_tiles_max, int sms) {
  int s = pairs >= sms ? 1 : sms / pairs;
  int max_s = n_tiles_max / 2;
  if (max_s < 1) max_s = 1;
  if (max_s > 32) max_s = 32;
  return s < max_s ? s : max_s;
}

// Key ranges of the fp32 kernel per (sequence, KV head, row chunk): as many
// as two CTAs per SM allow, one range per kF32Granule keys at most, in a
// cluster size whose clusters the device holds all at once (a second wave
// doubles the time: B = 2, k = 8, 2048 keys, 16 jobs, measured with the
// 4-warp form 30.3 us at 12 ranges, 34.0 at 16, where 14 clusters fit).
static int f32_splits(const AttnPlan& p) {
  const F32Kernel kern = f32_kernel_for(p.D, p.M);
  const long long jobs = (long long)p.B * p.Hkv * ((p.M + kern.rows - 1) / kern.rows);
  const long long keys = (long long)p.Lmax + p.k;
  const long long by_keys = (keys + kF32Granule - 1) / kF32Granule;
  if (jobs <= 0) return 1;
  for (int s : {16, 12, 10, 8, 6, 5, 4, 3, 2}) {
    if (s > by_keys || s * jobs > 2ll * num_sms()) continue;
    if (cluster_slots(kern.fn, kern.threads, kern.smem, s) >= jobs) return s;
  }
  return 1;
}

AttnPlan attn_plan(const sbd_attn_desc& d) {
  AttnPlan p;
  p.B = d.batch;
  p.k = d.block_k;
  p.Hq = d.n_q_heads;
  p.Hkv = d.n_kv_heads;
  p.G = d.n_q_heads / d.n_kv_heads;
  p.D = d.head_dim;
  p.Lmax = d.max_cache_len;
  p.M = p.G * p.k;
  p.bf16 = d.dtype == SBD_DTYPE_BF16;
  p.n_causal = 0;
  const float scale = d.scale != 0.f ? d.scale : 1.0f / sqrtf((float)d.head_dim);
  p.scale_log2 = scale * kLog2e;
  const int tiles = (p.Lmax + kTileKeys - 1) / kTileKeys + 1;
  if (!p.bf16) {
    p.splits = f32_splits(p);
  } else if (d.num_splits > 0) {
    p.splits = d.num_splits;
  } else {
    p.splits = choose_splits(p.B * p.Hkv, tiles, num_sms());
  }
  p.wide = p.bf16 && p.M > 64;
  // tcgen05 path: the splits of a (sequence, KV head) merge in shared memory
  // as one thread-block cluster (at most 16 CTAs) when the device can hold
  // all the clusters at once.  An automatic split count is lowered, down to
  // 3/5 of it, to the largest cluster size that fits (GB300, one 227 KB CTA
  // per SM: 36 clusters of 4, 15 of 8, 7 of 16); at batch 1, Llama-8B, 4096
  // cached keys, 12 splits in clusters took 12.9 us against 13.9 us for 19
  // splits merged by attn_combine_kernel.  Otherwise the partials go through
  // the workspace and attn_combine_kernel.
  p.cluster = !p.bf16 && p.splits > 1;
  if (p.bf16 && p.B > 0 && p.splits >= 2) {
    const int hi = p.splits < 16 ? p.splits : 16;
    const int lo = d.num_splits > 0 ? p.splits : (3 * p.splits + 4) / 5;
    for (int s = hi; s >= lo && s >= 2; --s) {
      if (attn_tc_cluster_ok(p, s)) {
        p.splits = s;
        p.cluster = true;
        break;
      }
    }
  }
  // The kernel by the keys of a CTA; both hold the same clusters (one 227 KB
  // CTA per SM), else the choice stays.
  if (p.bf16 && !p.wide) {
    p.wide = attn_use_wide(p);
    if (p.wide && p.cluster && !attn_tc_cluster_ok(p, p.splits)) p.wide = false;
  }
  // With more CTAs than one wave, the CTAs take the sequences longest first
  // (the pick costs B^2 comparisons per CTA, hence the batch limit).
  p.order = p.bf16 && p.B > 1 && p.B <= kOrderMaxB &&
            (long long)p.B * p.Hkv * p.splits > num_sms();
  return p;
}

size_t attn_workspace_bytes(const AttnPlan& p) {
  if (p.splits <= 1 || p.cluster) return 0;
  const size_t n = (size_t)p.B * p.Hkv * p.splits * p.M;
  return align_up(n * p.D * sizeof(float), 256) + align_up(n * sizeof(float), 256);
}

sbd_status attn_launch(const AttnPlan& p, const void* q, const void* kc, const void* vc,
                       const int32_t* lens, const void* kb, const void* vb, void* out, void* ws,
                       void* kc_app, void* vc_app, cudaStream_t st) {
  if (p.B == 0) return SBD_OK;
  int* err = device_error_word();
  if (!p.bf16) {
    F32Args a;
    a.q = (const float*)q;
    a.kc = (const float*)kc;
    a.vc = (const float*)vc;
    a.lens = lens;
    a.kb = (const float*)kb;
    a.vb = (const float*)vb;
    a.out = (float*)out;
    a.err = err;
    a.kc_app = (float*)kc_app;
    a.vc_app = (float*)vc_app;
    a.k = p.k;
    a.Hq = p.Hq;
    a.Hkv = p.Hkv;
    a.G = p.G;
    a.M = p.M;
    a.Lmax = p.Lmax;
    a.n_causal = p.n_causal;
    a.splits = p.splits;
    a.scale_log2 = p.scale_log2;
    const F32Kernel kern = f32_kernel_for(p.D, p.M);
    a.chunks = (p.M + kern.rows - 1) / kern.rows;
    const sbd_status s = allow_smem(kern.fn, kern.smem, "cudaFuncSetAttribute(attn_f32_kernel)");
    if (s != SBD_OK) return s;
    void* args[] = {(void*)&a};
    return launch_pdl(kern.fn, dim3(p.splits, p.Hkv * a.chunks, p.B), dim3(kern.threads),
                      kern.smem, st, args, "attn_f32_kernel launch", p.splits);
  }

  // 4-D tensor maps over the caches: dims (D, Hkv, Lmax, B), 64x64 boxes.
  CUtensorMap tk, tv;
  const uint64_t dims[4] = {(uint64_t)p.D, (uint64_t)p.Hkv, (uint64_t)p.Lmax, (uint64_t)p.B};
  const uint64_t strides[3] = {(uint64_t)p.D * 2, (uint64_t)p.Hkv * p.D * 2,
                               (uint64_t)p.Lmax * p.Hkv * p.D * 2};
  const uint32_t box[4] = {64, 1, (uint32_t)kTileKeys, 1};
  sbd_status s = encode_tensor_map(&tk, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void*)kc, dims,
                                   strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
  if (s != SBD_OK) return s;
  s = encode_tensor_map(&tv, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void*)vc, dims, strides, box,
                        CU_TENSOR_MAP_SWIZZLE_128B);
  if (s != SBD_OK) return s;

  // partials of a split that does not merge inside a cluster
  const size_t n = (size_t)p.B * p.Hkv * p.splits * p.M;
  const bool use_ws = p.splits > 1 && !p.cluster;
  float* part_o = use_ws ? (float*)ws : nullptr;
  float* part_lse = use_ws ? (float*)((char*)ws + align_up(n * p.D * sizeof(float), 256)) : nullptr;

  // Every bf16 shape runs on the tcgen05 kernels (block_attention_tc.cu).
  // Up to 16 packed rows a mma.sync kernel had measured faster than the
  // first tcgen05 form; against the current one it lost at every row count
  // (16 rows, batch 16, KV 8192: 91.2 against 88.9 us; batch 1, KV 4096,
  // 4 rows: 25.4 against 21.3 us) and was removed.
  s = attn_tc_launch(p, tk, tv, q, lens, kb, vb, out, part_o, part_lse, kc_app, vc_app, st);
  if (s != SBD_OK) return s;
  if (use_ws) {
    const float* po = part_o;
    const float* pl = part_lse;
    __nv_bfloat16* o = (__nv_bfloat16*)out;
    int k = p.k, Hq = p.Hq, Hkv = p.Hkv, G = p.G, M = p.M, S = p.splits;
    void* args[] = {(void*)&po, (void*)&pl, (void*)&o, (void*)&k, (void*)&Hq, (void*)&Hkv,
                    (void*)&G,  (void*)&M,  (void*)&S};
    const void* fn = p.D == 128 ? (const void*)attn_combine_kernel<128, __nv_bfloat16>
                                : (const void*)attn_combine_kernel<64, __nv_bfloat16>;
    s = launch_pdl(fn, dim3((p.M + kCombineRows - 1) / kCombineRows, p.Hkv, p.B),
                   dim3(32 * kCombineRows), 0, st, args, "attn_combine_kernel launch");
    if (s != SBD_OK) return s;
  }
  return SBD_OK;
}

}  // namespace sbd
