// Shared pieces of the bf16 LM-head kernels on the 5th-generation tensor
// cores (pair_lse.cu, pair_bwd_image.cu, pair_bwd_cluster.cu) and of their
// host orchestration (pair_grad_tc.cu): the warp-specialised CTA shape,
// small device helpers, tensor-map and grid helpers, and the entry points of
// each stage.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "pair_common.cuh"
#include "tc_ptx.cuh"

namespace pairk {
namespace tck {

using namespace tc;

// CTA of the head kernels: warp 0 = TMA producer, warp 1 = TMEM owner and
// single-thread MMA issuer, warps 2..5 = epilogue (one TMEM lane quadrant
// each, one tile row per thread).
constexpr int kThreads = 192;
constexpr int kAtom128 = 128 * 64 * 2;  // 128 rows x 64 bf16 (16 KB)
constexpr int kAllBlocks = 0x7fffffff;  // "every token block" for chunked passes

// Named barrier of the four epilogue warps (128 threads).
__device__ __forceinline__ void epi_sync() {
  asm volatile("bar.sync 1, 128;" ::: "memory");
}

__device__ __forceinline__ uint8_t *align1k(uint8_t *p) {
  return reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(p) + 1023) &
                                     ~static_cast<uintptr_t>(1023));
}

// Bulk copy global -> this CTA's shared memory, completing on `bar`.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes,
                                          uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes "
      "[%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Bulk copy of `bytes` (multiple of 16, both addresses 16-byte aligned) from
// this CTA's shared memory to global memory, tracked by this thread's bulk
// groups, with an L2 evict-first hint.
__device__ __forceinline__ void bulk_store_evict_first(void *dst, const void *src,
                                                       uint32_t bytes) {
  asm volatile(
      "{\n\t.reg .b64 pol;\n\t"
      "createpolicy.fractional.L2::evict_first.b64 pol, 1.0;\n\t"
      "cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, pol;\n\t}" ::"l"(
          reinterpret_cast<uint64_t>(dst)),
      "r"(smem_u32(src)), "r"(bytes)
      : "memory");
}

// <h, w> over d bf16 elements by one warp (d a multiple of 8, rows 16-byte
// aligned): fp32 sums of the products in a fixed order (lane-strided
// 8-element pieces, then the warp's butterfly); every lane gets the sum.
__device__ __forceinline__ float target_logit_dot(int d, const __nv_bfloat16 *h,
                                                  const __nv_bfloat16 *w, int lane) {
  float acc = 0.f;
  for (int k = lane * 8; k < d; k += 256) {
    const uint4 hu = *reinterpret_cast<const uint4 *>(h + k);
    const uint4 wu = *reinterpret_cast<const uint4 *>(w + k);
    const __nv_bfloat162 *hb = reinterpret_cast<const __nv_bfloat162 *>(&hu);
    const __nv_bfloat162 *wb = reinterpret_cast<const __nv_bfloat162 *>(&wu);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 hf = __bfloat1622float2(hb[i]), wf = __bfloat1622float2(wb[i]);
      acc = fmaf(hf.x, wf.x, acc);
      acc = fmaf(hf.y, wf.y, acc);
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}

__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// Work list of the persistent backward kernels (dh_gemm_kernel,
// dw_gemm_kernel, bwd_kernel): the units that fill whole rounds of the grid (ncl
// clusters or CTAs) run over all of their K extent; the R < ncl units left over are
// cut into S parts of K each, which run in as many rounds as they need. Of
// hidden sizes whose last unit per row block is 256 columns wide (every nq-th of
// all units), these take half the time and get Sh = ceil(S / 2) parts. Work item
// i < full_end is unit i; then come parts 0 .. Sh - 1 of all R units, then
// parts Sh .. S - 1 of the wide ones, part-major: the units that read the same
// rows of the K-indexed operand in a part run next to each other and share them
// in L2. Part p covers K steps [p nks / P, (p + 1) nks / P) of its unit's P. The
// item's fp32 tile goes to the scratch slot of its place in the list and the
// kernel's tail-combine pass adds a unit's parts in order (deterministic).
//
// S is the count of the smallest makespan, rounds x (steps of a part +
// overhead) + the combine pass's share per tile, of up to 64 and up to the
// scratch's `cap` tiles; S = 1 needs none. One round of S = ncl / R parts
// leaves up to half of the clusters idle: 55 units on 76 clusters in one part
// each take 2374 steps of 64 vocabulary rows, in four 3 x 594 (d = 2560, 11
// token pairs: 1321 and 1093 us). (Equal contiguous ranges of all R nks steps, one
// per cluster, leave none idle but read each W row at R different times:
// 1.35 times as slow as whole parts, from DRAM.)
struct TailSplit {
  int full_end, R, S, Sh;
  int Rh, h0, nq;  // narrow units among the R: at h0, h0 + nq, ...

  __device__ __forceinline__ int items() const { return R * Sh + (R - Rh) * (S - Sh); }
  __device__ __forceinline__ bool narrow(int v) const {
    return Rh > 0 && v >= h0 && (v - h0) % nq == 0;
  }
  __device__ __forceinline__ int parts(int v) const { return narrow(v) ? Sh : S; }
  // The j-th wide unit, and the number of wide ones before unit v.
  __device__ __forceinline__ int wide_at(int j) const {
    return j < h0 ? j : j + 1 + (j - h0) / (nq - 1);
  }
  __device__ __forceinline__ int wide_before(int v) const {
    return v > h0 ? v - 1 - (v - 1 - h0) / nq : v;
  }
};
constexpr int kTailMaxParts = 64;
// A whole warp calls (every lane gets the answer). d gives the units' widths (a
// multiple of 512: all alike); `tile` is the combine pass's share per scratch tile
// in 1/64 steps; own: the units' first parts need no scratch (slots R and up).
__device__ __forceinline__ TailSplit tail_split(int n_units, int ncl, int cap, int nks,
                                                int overhead, int tile, int d, bool own = false) {
  TailSplit t{n_units, 0, 1, 1, 0, 0, (d + 511) / 512};
  const int R = n_units % ncl;
  if (R == 0 || nks == 0) return t;
  t.R = R;
  t.h0 = t.nq - 1 - (n_units - R) % t.nq;
  if (t.nq > 1 && d % 512 != 0 && d % 512 <= 256 && R > t.h0)
    t.Rh = 1 + (R - 1 - t.h0) / t.nq;
  unsigned long long best = ~0ull;
  for (int S = 1 + (threadIdx.x & 31); S <= min(kTailMaxParts, nks); S += 32) {
    t.S = S;
    t.Sh = t.Rh > 0 ? (S + 1) / 2 : S;
    const int n = t.items();
    if (S > 1 && n - (own ? R : 0) > cap) break;
    const long long rounds = (n + ncl - 1) / ncl, steps = (nks + S - 1) / S;
    const long long cost = 64 * rounds * (steps + overhead) + (S > 1 ? (long long)tile * n : 0);
    best = min(best, (unsigned long long)cost * (2 * kTailMaxParts) + S);
  }
  for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
  t.S = (int)(best % (2 * kTailMaxParts));
  t.Sh = t.Rh > 0 ? (t.S + 1) / 2 : t.S;
  if (t.S < 2) return TailSplit{n_units, 0, 1, 1, 0, 0, t.nq};
  t.full_end = n_units - R;
  return t;
}
// Work item i of a TailSplit -> unit u, its K steps [k0, k1) and scratch
// slot (-1: a whole unit).
__device__ __forceinline__ void tail_item(const TailSplit &tl, int nks, int i, int &u, int &k0,
                                          int &k1, int &slot) {
  if (i < tl.full_end) {
    u = i; k0 = 0; k1 = nks; slot = -1;
  } else {
    const int j = i - tl.full_end, all = tl.R * tl.Sh, wide = tl.R - tl.Rh;
    int part, v;
    if (j < all) {
      part = j / tl.R;
      v = j - part * tl.R;
    } else {
      part = (j - all) / wide;
      v = tl.wide_at(j - all - part * wide);
      part += tl.Sh;
    }
    const int parts = tl.parts(v);
    u = tl.full_end + v;
    k0 = (int)((int64_t)part * nks / parts);
    k1 = (int)((int64_t)(part + 1) * nks / parts);
    slot = j;
  }
}
// First part `acc` of unit full_end + v plus its others at float4 `at` of their
// tiles (`tile` float4 each, the second part's being `src`), in part order; eight
// loads in flight.
__device__ __forceinline__ float4 tail_sum(const TailSplit &tl, int v, float4 acc,
                                           const float4 *src, int64_t tile, int64_t at) {
  auto add = [&](const float4 *p, int64_t stride, int n) {
    int k = 0;
    for (; k + 8 <= n; k += 8, p += 8 * stride) {
      float4 x[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) x[q] = p[q * stride];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        acc.x += x[q].x; acc.y += x[q].y; acc.z += x[q].z; acc.w += x[q].w;
      }
    }
    for (; k < n; ++k, p += stride) {
      const float4 x = *p;
      acc.x += x.x; acc.y += x.y; acc.z += x.z; acc.w += x.w;
    }
  };
  add(src + at, tl.R * tile, tl.Sh - 1);
  if (!tl.narrow(v))
    add(src + ((int64_t)tl.R * (tl.Sh - 1) + tl.wide_before(v) - v) * tile + at,
        (tl.R - tl.Rh) * tile, tl.S - tl.Sh);
  return acc;
}

// ---- host helpers (pair_grad_tc.cu)
PFN_cuTensorMapEncodeTiled_v12000 encode_fn();
// 2-D bf16 row-major [rows][cols] map with 64 x box_rows SWIZZLE_128B boxes.
bool make_map(CUtensorMap *m, const void *ptr, int64_t rows, int64_t cols, int box_rows);
// 2-D fp32 row-major [rows][cols] map with 32 x 32 SWIZZLE_128B boxes (stores).
bool make_map_f32(CUtensorMap *m, const void *ptr, int64_t rows, int64_t cols);
// 3-D bf16 map: dims (innermost first), byte strides of dims 1 and 2, box, swizzle.
bool make_map3(CUtensorMap *m, const void *ptr, const cuuint64_t (&dims)[3],
               const cuuint64_t (&strides)[2], const cuuint32_t (&box)[3],
               CUtensorMapSwizzle sw);
int num_sms();
// CTAs of a persistent grid of 2-CTA clusters (occupancy API; cached in *cache).
int pair_grid(const void *kernel, size_t smem, int *cache);

// ---- stages of the head
// Log-sum-exp pass over token blocks [rb0, rb0 + cap), then lse of those
// tokens. With image, the softmax terms are taken relative to the reference
// (rows_kernel, pair_grad_prep.cu), the bf16 terms of its first s_blocks blocks are kept as
// the image, and rows too far above their reference are redone (pair_lse.cu).
pair_status launch_lse(const GradArgs &g, const GradWorkspace &w, cudaStream_t s, int rb0,
                       int cap, bool image, int s_blocks);
// One token chunk of the image backward: scaled hidden rows, dh_gemm,
// dw_gemm (pair_bwd_image.cu).
pair_status launch_chunk_bwd(const GradArgs &g, const GradWorkspace &w, cudaStream_t s,
                             int64_t c);
// Gradient tiles of token blocks x vocabulary tiles (pair_lse.cu), and the
// backward that uses them where the workspace holds no image
// (pair_bwd_image.cu).
pair_status launch_grad_image(const GradArgs &g, const GradWorkspace &w, cudaStream_t s, int rb0,
                              int cap, int tile0, int n_vt, void *img);
pair_status grad_bwd_slabs(const GradArgs &g, const GradWorkspace &w, cudaStream_t s, bool &dh,
                           bool &dw);
// Backward without an image, recomputing the logits (pair_bwd_cluster.cu), and
// what one of its products takes where no cluster form applies.
double bwd_recompute_us(int d, double rows, double cols, int64_t rows_max, int64_t cols_max,
                        size_t scratch_bytes);
pair_status grad_bwd_recompute(const GradArgs &g, const GradWorkspace &w, cudaStream_t s);
// Whole head without an image: fused log-sum-exp + dH, then dW (cluster
// form; d = 512 A, A <= 6). lse, zy and dH, dW softmax parts as the
// three-pass sequence leaves them.
bool onchip_fused_applies(int d);
pair_status grad_head_onchip(const GradArgs &g, const GradWorkspace &w, cudaStream_t s);

inline bool image_path(const GradWorkspace &w) { return w.gimg && w.hs && w.gimg_rb > 0; }
inline int64_t image_chunks(const GradArgs &g, const GradWorkspace &w) {
  return ((g.T + 127) / 128 + w.gimg_rb - 1) / w.gimg_rb;
}

}  // namespace tck
}  // namespace pairk
