// pair_grad bookkeeping kernels: active-token compaction, per-rollout and
// total objective, exact one-hot gradient parts, workspace layout.
//
// The objective of Sec. 4.5 is sum_i a_i log pi(o_i | q) with log pi a sum
// over response tokens; rollouts with a_i == 0 contribute nothing and are
// removed before any head arithmetic. The surviving tokens are packed in
// their original order (rollout by rollout), so every per-rollout sum below
// runs over a contiguous range in a fixed order (bit-reproducible).
#include <cuda_bf16.h>

#include "pair_common.cuh"

namespace pairk {
namespace {

constexpr int kNSplit = 16;  // vocabulary splits of the log-sum-exp pass
constexpr int kTicket = 3;   // counters[]: blocks of finalize_kernel that are done

__device__ __forceinline__ bool coef_nonzero(float a) {
  return (__float_as_uint(a) & 0x7fffffffu) != 0u;
}

__device__ __forceinline__ int clamp_i(int v, int lo, int hi) {
  return v < lo ? lo : (v > hi ? hi : v);
}

// Counts the active tokens of each rollout; validates every mask=1 target.
// Clears the one-hot part's n_bkt bucket counters and the finalize ticket.
__global__ void seg_count_kernel(int R, int T, int V, const int32_t *cu,
                                 const uint8_t *mask, const int32_t *y,
                                 const float *a, int32_t *seg_cnt, int32_t *counters,
                                 int32_t *bkt, int n_bkt, int32_t *dev_err) {
  const int i = blockIdx.x;
  if (i == 0 && threadIdx.x == 0) counters[kTicket] = 0;
  for (int k = i * blockDim.x + threadIdx.x; k < n_bkt; k += gridDim.x * blockDim.x) bkt[k] = 0;
  const int beg = clamp_i(cu[i], 0, T), end = clamp_i(cu[i + 1], beg, T);
  const bool on = coef_nonzero(a[i]);
  int n = 0, bad = 0;
  for (int t = beg + threadIdx.x; t < end; t += blockDim.x) {
    if (mask[t]) {
      ++n;
      const int yt = y[t];
      bad |= (yt < 0 || yt >= V);
    }
  }
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  __shared__ int red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = n;
  if (bad) flag_error(dev_err, PAIR_DEV_ERR_TARGET_RANGE);
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[k];
    seg_cnt[i] = on ? s : 0;
  }
}

// Exclusive prefix over rollouts (one block, sequential chunks of 1024), for
// more than kGatherScanMax of them.
__global__ void seg_scan_kernel(int R, const int32_t *seg_cnt, int32_t *seg_off,
                                int32_t *counters) {
  __shared__ int buf[1024];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < R; base += 1024) {
    const int i = base + threadIdx.x;
    const int v = i < R ? seg_cnt[i] : 0;
    buf[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
      const int add = threadIdx.x >= o ? buf[threadIdx.x - o] : 0;
      __syncthreads();
      buf[threadIdx.x] += add;
      __syncthreads();
    }
    if (i < R) seg_off[i] = carry + buf[threadIdx.x] - v;
    __syncthreads();
    if (threadIdx.x == 1023) carry += buf[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    seg_off[R] = carry;
    counters[0] = carry;
  }
}

// Rollouts up to which gather_kernel's blocks each sum the counts before their
// own (a few coalesced loads, instead of a launch of its own for the scan).
constexpr int kGatherScanMax = 2048;

// In-order compaction of each active rollout's mask=1 tokens; with `sum` also
// the rollout offsets and the total. Targets out of range (reported by
// seg_count) are taken as 0, so that no later kernel reads past W. Counts the
// tokens per target bucket in cnt (nullable).
__global__ void __launch_bounds__(1024)
    gather_kernel(int R, int T, int V, const int32_t *cu, const uint8_t *mask, const int32_t *y,
                  const float *a, const int32_t *seg_cnt, bool sum, int32_t *seg_off,
                  int32_t *counters, int32_t *tok_idx, int32_t *tok_y, float *tok_c,
                  int32_t *cnt) {
  const int i = blockIdx.x;
  __shared__ int wsum[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  int carry;
  if (sum) {
    int n = 0;
    for (int k = threadIdx.x; k < i; k += blockDim.x) n += seg_cnt[k];
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) wsum[w] = n;
    __syncthreads();
    carry = __reduce_add_sync(0xffffffffu, lane < nw ? wsum[lane] : 0);
    __syncthreads();
    if (threadIdx.x == 0) {
      seg_off[i] = carry;
      if (i == R - 1) seg_off[R] = counters[0] = carry + seg_cnt[i];
    }
  } else {
    carry = seg_off[i];
  }
  const float c = a[i];
  if (!coef_nonzero(c)) return;
  const int beg = clamp_i(cu[i], 0, T), end = clamp_i(cu[i + 1], beg, T);
  for (int base = beg; base < end; base += blockDim.x) {
    const int t = base + threadIdx.x;
    const int f = (t < end && mask[t]) ? 1 : 0;
    const unsigned bal = __ballot_sync(0xffffffffu, f);
    const int rank_w = __popc(bal & ((1u << lane) - 1u));
    if (lane == 0) wsum[w] = __popc(bal);
    __syncthreads();
    const int mine = lane < nw ? wsum[lane] : 0;
    const int before = __reduce_add_sync(0xffffffffu, lane < w ? mine : 0);
    const int total = __reduce_add_sync(0xffffffffu, mine);
    if (f) {
      const int p = carry + before + rank_w;
      int yt = y[t];
      if (yt < 0 || yt >= V) yt = 0;
      tok_idx[p] = t;
      tok_y[p] = yt;
      tok_c[p] = c;
      if (cnt) atomicAdd(&cnt[yt / kOneHotBucket], 1);
    }
    carry += total;
    __syncthreads();
  }
}

constexpr int kZeroCuSmem = 8192;  // rollout offsets staged in shared memory, at most

// One warp per row, two independent parts:
// - Hc[p] = H[tok_idx[p]] for p < T_eff, and zero rows up to the next multiple
//   of 128 (the token-tile height), so tail tiles carry finite zeros. With ref,
//   the reference of the image path's log-sum-exp pass from the same loads:
//   ref[p] = <h, W[y]> log2 e, fp32 sums of the products in a fixed order
//   (lane-strided 8-element pieces, then the warp's butterfly).
// - the dH rows of tokens outside the objective (mask = 0 or a = 0) are zeroed.
// As three kernels (copy, zero, reference) this took 8 us more per call at 1.3
// k tokens and read Hc once more.
template <typename Tin>
__global__ void __launch_bounds__(256)
    rows_kernel(int64_t T, int64_t Tpad, int d, int R, const int32_t *counters,
                const int32_t *tok_idx, const int32_t *tok_y, const Tin *H, const Tin *W,
                Tin *Hc, float *ref, const int32_t *cu, const uint8_t *mask, const float *a,
                float *dH) {
  // The rollout offsets are searched once per row by every lane: from shared
  // memory when they fit, so the search costs no global round trips.
  extern __shared__ int32_t cu_s[];
  const bool staged = R + 1 <= kZeroCuSmem;
  if (staged)
    for (int i = threadIdx.x; i <= R; i += blockDim.x) cu_s[i] = cu[i];
  __syncthreads();
  const int32_t *cs = staged ? cu_s : cu;
  const int lane = threadIdx.x & 31;
  const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;

  const int Teff = counters[0];
  const int64_t Tz = min(((int64_t)Teff + 127) / 128 * 128, Tpad);
  constexpr int kVec = 16 / (int)sizeof(Tin);
  const int dv = d / kVec;
  for (int64_t p = w0; p < Tz; p += nw) {
    uint4 *dst = reinterpret_cast<uint4 *>(Hc + p * d);
    if (p >= Teff) {
      for (int k = lane; k < dv; k += 32) dst[k] = make_uint4(0u, 0u, 0u, 0u);
      continue;
    }
    const uint4 *src = reinterpret_cast<const uint4 *>(H + (int64_t)tok_idx[p] * d);
    if (sizeof(Tin) == 2 && ref) {
      const uint4 *wr = reinterpret_cast<const uint4 *>(W + (int64_t)tok_y[p] * d);
      float acc = 0.f;
#pragma unroll 4
      for (int k = lane; k < dv; k += 32) {
        const uint4 hu = src[k], wu = wr[k];
        dst[k] = hu;
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
      if (lane == 0) ref[p] = acc * kLog2e;
    } else {
#pragma unroll 4
      for (int k = lane; k < dv; k += 32) dst[k] = src[k];
    }
  }

  for (int64_t t = w0; t < T; t += nw) {
    // rollout of t: last i with cu[i] <= t
    int lo = 0, hi = R - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (cs[mid] <= t) lo = mid; else hi = mid - 1;
    }
    const bool live = mask[t] && coef_nonzero(a[lo]) && cs[lo] <= t && t < cs[lo + 1];
    if (live) continue;
    float4 *row = reinterpret_cast<float4 *>(dH + t * d);  // d is a multiple of 16
    for (int k = lane; k < d / 4; k += 32) row[k] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// Sum of logp_t = zy - lse over a rollout's compacted range (fp64, fixed tree
// order), by a block; the result in thread 0.
__device__ double seg_logp_sum(int beg, int end, const float *zy, const float *lse) {
  double s = 0.0;
  for (int p = beg + threadIdx.x; p < end; p += blockDim.x) s += (double)zy[p] - (double)lse[p];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ double red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[k];
  return t;
}

// Per-rollout log-probabilities, and by the last block to finish the
// objective Jobj = sum_i a_i * logp_seq_i (fp64, fixed order); logp_seq out.
__global__ void __launch_bounds__(256)
    finalize_kernel(int R, const int32_t *seg_off, const float *zy, const float *lse,
                    const float *a, double *seg_logp, int32_t *counters, double *Jobj,
                    float *logp_seq) {
  const int i = blockIdx.x;
  const double lp_i = seg_logp_sum(seg_off[i], seg_off[i + 1], zy, lse);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    seg_logp[i] = lp_i;
    __threadfence();
    last = atomicAdd(&counters[kTicket], 1) == R - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  __shared__ double red[32];
  double s = 0.0;
  for (int k = threadIdx.x; k < R; k += blockDim.x) {
    const bool on = coef_nonzero(a[k]);
    const double lp = on ? __ldcg(seg_logp + k) : 0.0;
    if (logp_seq) logp_seq[k] = (float)lp;
    s += on ? (double)a[k] * lp : 0.0;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[k];
    *Jobj = t;
  }
}

// Eight consecutive elements as fp32.
__device__ __forceinline__ void load8(const __nv_bfloat16 *h, float (&x)[8]) {
  const uint4 u = *reinterpret_cast<const uint4 *>(h);
  const __nv_bfloat162 *b = reinterpret_cast<const __nv_bfloat162 *>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __bfloat1622float2(b[i]);
    x[2 * i] = f.x;
    x[2 * i + 1] = f.y;
  }
}
__device__ __forceinline__ void load8(const float *h, float (&x)[8]) {
  const float4 a = reinterpret_cast<const float4 *>(h)[0];
  const float4 b = reinterpret_cast<const float4 *>(h)[1];
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
  x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}

// dH_t += c_t W[y_t]  (the one-hot part of dJ/dh_t, exact in fp32): 8
// columns per thread with vector accesses (d is a multiple of 8 on both
// paths), two tokens in flight per block.
template <typename Tin>
__global__ void onehot_dh_kernel(int d, const int32_t *counters,
                                 const int32_t *tok_idx, const int32_t *tok_y,
                                 const float *tok_c, const Tin *W, float *dH) {
  const int Teff = counters[0];
  const int d8 = d / 8;
  for (int p0 = 2 * blockIdx.x; p0 < Teff; p0 += 2 * gridDim.x) {
    const bool two = p0 + 1 < Teff;
    const float c0 = tok_c[p0], c1 = two ? tok_c[p0 + 1] : 0.f;
    const Tin *w0 = W + (int64_t)tok_y[p0] * d;
    const Tin *w1 = two ? W + (int64_t)tok_y[p0 + 1] * d : w0;
    float *r0 = dH + (int64_t)tok_idx[p0] * d;
    float *r1 = two ? dH + (int64_t)tok_idx[p0 + 1] * d : r0;
    for (int k8 = threadIdx.x; k8 < d8; k8 += blockDim.x) {
      const int k = 8 * k8;
      float x0[8], x1[8];
      load8(w0 + k, x0);
      float4 a0 = reinterpret_cast<float4 *>(r0 + k)[0];
      float4 b0 = reinterpret_cast<float4 *>(r0 + k)[1];
      float4 a1 = a0, b1 = b0;
      if (two) {
        load8(w1 + k, x1);
        a1 = reinterpret_cast<float4 *>(r1 + k)[0];
        b1 = reinterpret_cast<float4 *>(r1 + k)[1];
      }
      reinterpret_cast<float4 *>(r0 + k)[0] =
          make_float4(fmaf(c0, x0[0], a0.x), fmaf(c0, x0[1], a0.y), fmaf(c0, x0[2], a0.z),
                      fmaf(c0, x0[3], a0.w));
      reinterpret_cast<float4 *>(r0 + k)[1] =
          make_float4(fmaf(c0, x0[4], b0.x), fmaf(c0, x0[5], b0.y), fmaf(c0, x0[6], b0.z),
                      fmaf(c0, x0[7], b0.w));
      if (two) {
        reinterpret_cast<float4 *>(r1 + k)[0] =
            make_float4(fmaf(c1, x1[0], a1.x), fmaf(c1, x1[1], a1.y), fmaf(c1, x1[2], a1.z),
                        fmaf(c1, x1[3], a1.w));
        reinterpret_cast<float4 *>(r1 + k)[1] =
            make_float4(fmaf(c1, x1[4], b1.x), fmaf(c1, x1[5], b1.y), fmaf(c1, x1[6], b1.z),
                        fmaf(c1, x1[7], b1.w));
      }
    }
  }
}

// dW_v += sum_{t: y_t = v} c_t h_t (the one-hot part of dJ/dW_v), exact in
// fp32, tokens added in their packed order. The compacted tokens are grouped
// by target bucket (kOneHotBucket vocabulary rows): counts, offsets and a
// fill (in any order); then one warp owns a bucket and puts its tokens in
// packed order: up to 32 by a bitonic sort in registers, up to
// kOneHotRankMax by ranking each against all others into shared memory; a
// heavier bucket instead scans the compacted targets in order for its rows
// (four 32-token chunks per round, so the target loads overlap). A row is
// updated with 16-byte vector accesses when d allows it.
template <typename Tin>
__device__ __forceinline__ void axpy_row(int d, float c, const Tin *__restrict__ h,
                                         float *__restrict__ row, int lane) {
  if ((d & 7) == 0) {
    for (int k0 = lane * 8; k0 < d; k0 += 32 * 8 * 2) {
      // Two independent 8-element groups per iteration.
      const int k1 = k0 + 32 * 8;
      float x0[8], x1[8];
      load8(h + k0, x0);
      float4 r0a = reinterpret_cast<float4 *>(row + k0)[0];
      float4 r0b = reinterpret_cast<float4 *>(row + k0)[1];
      float4 r1a = make_float4(0.f, 0.f, 0.f, 0.f), r1b = r1a;
      const bool has1 = k1 < d;
      if (has1) {
        load8(h + k1, x1);
        r1a = reinterpret_cast<float4 *>(row + k1)[0];
        r1b = reinterpret_cast<float4 *>(row + k1)[1];
      }
      r0a = make_float4(fmaf(c, x0[0], r0a.x), fmaf(c, x0[1], r0a.y), fmaf(c, x0[2], r0a.z),
                        fmaf(c, x0[3], r0a.w));
      r0b = make_float4(fmaf(c, x0[4], r0b.x), fmaf(c, x0[5], r0b.y), fmaf(c, x0[6], r0b.z),
                        fmaf(c, x0[7], r0b.w));
      reinterpret_cast<float4 *>(row + k0)[0] = r0a;
      reinterpret_cast<float4 *>(row + k0)[1] = r0b;
      if (has1) {
        r1a = make_float4(fmaf(c, x1[0], r1a.x), fmaf(c, x1[1], r1a.y), fmaf(c, x1[2], r1a.z),
                          fmaf(c, x1[3], r1a.w));
        r1b = make_float4(fmaf(c, x1[4], r1b.x), fmaf(c, x1[5], r1b.y), fmaf(c, x1[6], r1b.z),
                          fmaf(c, x1[7], r1b.w));
        reinterpret_cast<float4 *>(row + k1)[0] = r1a;
        reinterpret_cast<float4 *>(row + k1)[1] = r1b;
      }
    }
  } else {
    for (int k = lane; k < d; k += 32) row[k] = fmaf(c, (float)h[k], row[k]);
  }
}

// off[b] = sum of cnt[< b] for b <= nb (one block of 1024 threads, each over a
// contiguous run of buckets).
__global__ void __launch_bounds__(1024) onehot_scan_kernel(int nb, const int32_t *cnt,
                                                           int32_t *off) {
  __shared__ int32_t wsum[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (nb + 1024) / 1024;  // of nb + 1 offsets
  const int b0 = threadIdx.x * per, b1 = min(b0 + per, nb + 1);
  int v = 0;
#pragma unroll 8
  for (int b = b0; b < b1; ++b) v += b < nb ? cnt[b] : 0;
  int x = v;  // inclusive warp scan
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  int run = __reduce_add_sync(0xffffffffu, lane < warp ? wsum[lane] : 0) + x - v;
#pragma unroll 8
  for (int b = b0; b < b1; ++b) {
    off[b] = run;
    run += b < nb ? cnt[b] : 0;
  }
}

__global__ void onehot_fill_kernel(const int32_t *counters, const int32_t *tok_y,
                                   const int32_t *off, int32_t *fill, int32_t *blist) {
  const int Teff = counters[0];
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < Teff; p += gridDim.x * blockDim.x) {
    const int b = tok_y[p] / kOneHotBucket;
    blist[off[b] + atomicAdd(&fill[b], 1)] = p;
  }
}

// row += c h over d elements by 8 lanes (lane8 = lane index within them).
template <typename Tin>
__device__ __forceinline__ void axpy_row8(int d, float c, const Tin *__restrict__ h,
                                          float *__restrict__ row, int lane8) {
  if ((d & 7) == 0) {
    for (int k0 = lane8 * 8; k0 < d; k0 += 64) {
      float x[8];
      load8(h + k0, x);
      float4 ra = reinterpret_cast<float4 *>(row + k0)[0];
      float4 rb = reinterpret_cast<float4 *>(row + k0)[1];
      ra = make_float4(fmaf(c, x[0], ra.x), fmaf(c, x[1], ra.y), fmaf(c, x[2], ra.z),
                       fmaf(c, x[3], ra.w));
      rb = make_float4(fmaf(c, x[4], rb.x), fmaf(c, x[5], rb.y), fmaf(c, x[6], rb.z),
                       fmaf(c, x[7], rb.w));
      reinterpret_cast<float4 *>(row + k0)[0] = ra;
      reinterpret_cast<float4 *>(row + k0)[1] = rb;
    }
  } else {
    for (int k = lane8; k < d; k += 8) row[k] = fmaf(c, (float)h[k], row[k]);
  }
}

// Adds the one-hot terms of tokens q_0 < q_1 < ... (packed positions, given
// by get(i), i < n) in that order per target row: four consecutive tokens at
// a time, 8 lanes each, when their four rows differ; one at a time otherwise.
template <typename Tin, typename Get>
__device__ __forceinline__ void onehot_apply_sorted(int d, int n, Get get, const int32_t *tok_y,
                                                    const float *tok_c, const Tin *Hc,
                                                    float *dW, int lane) {
  int i = 0;
  while (i < n) {
    if (i + 4 <= n) {
      const int q0 = get(i), q1 = get(i + 1), q2 = get(i + 2), q3 = get(i + 3);
      const int y0 = tok_y[q0], y1 = tok_y[q1], y2 = tok_y[q2], y3 = tok_y[q3];
      if (y0 != y1 && y0 != y2 && y0 != y3 && y1 != y2 && y1 != y3 && y2 != y3) {
        const int g = lane >> 3;
        const int q = g == 0 ? q0 : g == 1 ? q1 : g == 2 ? q2 : q3;
        const int y = g == 0 ? y0 : g == 1 ? y1 : g == 2 ? y2 : y3;
        axpy_row8(d, tok_c[q], Hc + (int64_t)q * d, dW + (int64_t)y * d, lane & 7);
        __syncwarp();
        i += 4;
        continue;
      }
    }
    const int q = get(i);
    axpy_row(d, tok_c[q], Hc + (int64_t)q * d, dW + (int64_t)tok_y[q] * d, lane);
    __syncwarp();
    ++i;
  }
}

constexpr int kOneHotRankMax = 512;  // bucket tokens ranked in shared memory, at most

template <typename Tin>
__global__ void __launch_bounds__(256)
    onehot_dw_kernel(int d, int V, int nb, const int32_t *counters, const int32_t *tok_y,
                     const float *tok_c, const int32_t *off, const int32_t *blist,
                     const Tin *Hc, float *dW) {
  __shared__ int32_t sorted[8][kOneHotRankMax];  // per warp of the block
  const int bk = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (bk >= nb) return;
  const int b0 = off[bk], n = off[bk + 1] - b0;
  if (n == 0) return;
  if (n > 32 && n <= kOneHotRankMax) {
    // Rank each token against all others of the bucket (positions are
    // distinct), then add them in rank order.
    int32_t *srt = sorted[threadIdx.x >> 5];
    for (int i = lane; i < n; i += 32) {
      const int p = blist[b0 + i];
      int rank = 0;
      for (int j = 0; j < n; ++j) rank += blist[b0 + j] < p ? 1 : 0;
      srt[rank] = p;
    }
    __syncwarp();
    onehot_apply_sorted(d, n, [&](int i) { return srt[i]; }, tok_y, tok_c, Hc, dW, lane);
    return;
  }
  if (n <= 32) {
    // Bitonic sort of the bucket's packed positions across the warp.
    int p = lane < n ? blist[b0 + lane] : 0x7fffffff;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
      for (int j = k >> 1; j > 0; j >>= 1) {
        const int q = __shfl_xor_sync(0xffffffffu, p, j);
        p = (((lane & j) == 0) == ((lane & k) == 0)) ? min(p, q) : max(p, q);
      }
    onehot_apply_sorted(
        d, n, [&](int i) { return __shfl_sync(0xffffffffu, p, i); }, tok_y, tok_c, Hc, dW, lane);
    return;
  }
  const int v0 = bk * kOneHotBucket;
  const int v1 = min(V, v0 + kOneHotBucket);
  const int Teff = counters[0];
  for (int base = 0; base < Teff; base += 128) {
    int yt[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int pp = base + 32 * i + lane;
      yt[i] = pp < Teff ? tok_y[pp] : -1;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      unsigned hit = __ballot_sync(0xffffffffu, yt[i] >= v0 && yt[i] < v1);
      while (hit) {
        const int src = __ffs(hit) - 1;
        hit &= hit - 1;
        const int q = base + 32 * i + src;
        const int v = __shfl_sync(0xffffffffu, yt[i], src);
        axpy_row(d, tok_c[q], Hc + (int64_t)q * d, dW + (int64_t)v * d, lane);
      }
    }
  }
}

// Clipped trajectory-ratio surrogate of the practical PPO epochs (Sec. 4.5,
// App. "Practical departures"): for rollout i with detached coefficient
// A_i = a_i and ratio rho_i = exp(logp_seq_i - logp_old_i),
//   L_i = min(rho_i A_i, clip(rho_i, 1 - eps, 1 + eps) A_i),
// and the gradient coefficient c_i = A_i rho_i where the unclipped term is the
// minimum (A_i > 0: rho_i <= 1 + eps; A_i < 0: rho_i >= 1 - eps), else 0.
// The ratio is formed in fp64 from the fp64 per-rollout log-probability.
// One block per rollout: its summed log-probability, its coefficient, and
// tok_c[p] = c_i for its compacted tokens p.
__global__ void __launch_bounds__(256)
    ppo_coef_kernel(int R, const int32_t *seg_off, const float *zy, const float *lse,
                    const float *a, const float *logp_old, float eps, double *seg_logp, float *c,
                    double *L, float *coef_out, float *tok_c) {
  const int i = blockIdx.x;
  const int beg = seg_off[i], end = seg_off[i + 1];
  const double lp = seg_logp_sum(beg, end, zy, lse);
  __shared__ float c_s;
  if (threadIdx.x == 0) {
    const double A = (double)a[i];
    float ci = 0.f;
    double li = 0.0;
    if (coef_nonzero(a[i])) {
      const double ratio = exp(lp - (double)logp_old[i]);
      const double lo = 1.0 - (double)eps, hi = 1.0 + (double)eps;
      const double clipped = ratio < lo ? lo : (ratio > hi ? hi : ratio);
      const double u = ratio * A, v = clipped * A;
      li = u < v ? u : v;
      const bool unclipped = A > 0.0 ? ratio <= hi : ratio >= lo;
      ci = unclipped ? (float)(A * ratio) : 0.f;
    }
    seg_logp[i] = lp;
    c[i] = ci;
    L[i] = li;
    if (coef_out) coef_out[i] = ci;
    c_s = ci;
  }
  __syncthreads();
  const float ci = c_s;
  for (int p = beg + threadIdx.x; p < end; p += blockDim.x) tok_c[p] = ci;
}

// Jobj = sum_i L_i (fp64, fixed order); logp_seq out as in finalize_kernel.
__global__ void ppo_objective_kernel(int R, const float *a, const double *seg_logp,
                                     const double *L, double *Jobj, float *logp_seq) {
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < R; i += blockDim.x) {
    const bool on = coef_nonzero(a[i]);
    if (logp_seq) logp_seq[i] = on ? (float)seg_logp[i] : 0.f;
    s += L[i];
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[k];
    *Jobj = t;
  }
}

// logp_tok[t] = 0 for every packed token (the scatter below then fills the
// active ones).
__global__ void zero_f32_kernel(int64_t n, float *x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    x[i] = 0.f;
}

// logp_tok[tok_idx[p]] = zy[p] - lse[p] for every compacted token p.
__global__ void scatter_logp_kernel(const int32_t *counters, const int32_t *tok_idx,
                                    const float *zy, const float *lse, float *logp_tok) {
  const int Teff = counters[0];
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < Teff; p += gridDim.x * blockDim.x)
    logp_tok[tok_idx[p]] = zy[p] - lse[p];
}

}  // namespace

size_t grad_workspace_bytes(int64_t T, int32_t d, int32_t V, int32_t R,
                            pair_dtype dt, GradWorkspace *out, void *base, int gimg_rb) {
  const int64_t Tpad = (T + 127) / 128 * 128 + 128;
  const size_t esz = dt == PAIR_BF16 ? 2 : 4;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += (bytes + 255) / 256 * 256;
    return o;
  };
  const size_t o_cnt = take(64 * sizeof(int32_t));
  const size_t o_segc = take((size_t)R * 4);
  const size_t o_sego = take((size_t)(R + 1) * 4);
  const size_t o_idx = take((size_t)Tpad * 4);
  const size_t o_y = take((size_t)Tpad * 4);
  const size_t o_c = take((size_t)Tpad * 4);
  const size_t o_lse = take((size_t)Tpad * 4);
  const size_t o_zy = take((size_t)Tpad * 4);
  const size_t o_part = take((size_t)kNSplit * Tpad * sizeof(float2));
  const size_t o_segl = take((size_t)R * 8);
  const size_t o_ppoc = take((size_t)R * 4);
  const size_t o_ppol = take((size_t)R * 8);
  const size_t o_hc = take((size_t)Tpad * d * esz);
  const size_t nb = (size_t)((V + kOneHotBucket - 1) / kOneHotBucket);
  const size_t o_bkt = take(3 * (nb + 1) * 4);
  const size_t o_blist = take((size_t)Tpad * 4);
  const size_t o_ring = dt == PAIR_BF16 ? take((size_t)kMaxClusters * kRingBytesPerCluster) : off;
  const bool cl = dt == PAIR_BF16 && grad_cluster_path(d);
  // Hidden sizes the image backward takes (grad_gimg_rows): per-token
  // reference and softmax sum of its log-sum-exp pass.
  const bool img = dt == PAIR_BF16 && d >= 512 && d % 512 == 0;
  const size_t o_tail = cl ? take((size_t)kMaxClusters * 2 * 128 * d * sizeof(float)) : off;
  const int n_rbmax = (int)(Tpad / 128);
  const int n_slots = n_rbmax + 2 * kMaxClusters;
  const size_t o_ref = (cl || img) ? take((size_t)Tpad * 4) : off;
  const size_t o_mrow = (cl || img) ? take((size_t)Tpad * 4) : off;
  const size_t o_lsum = img ? take((size_t)Tpad * 4) : off;
  const size_t o_prog = img ? take((size_t)kMaxPairs * 4) : off;
  const size_t o_rbflag = cl ? take((size_t)n_rbmax * 4) : off;
  const size_t o_rblist = cl ? take((size_t)n_rbmax * 4) : off;
  const size_t o_ready = cl ? take((size_t)n_slots * 4) : off;
  const size_t o_lpart = cl ? take((size_t)n_slots * 8 * 256 * 4) : off;
  const size_t o_taill = cl ? take((size_t)kMaxClusters * 2 * 256 * 4) : off;
  // The image comes last, so that a larger workspace only adds token blocks.
  const size_t n_vt = (size_t)((V + 127) / 128);
  const size_t o_gimg = gimg_rb ? take((size_t)gimg_rb * n_vt * kGImgTileBytes) : off;
  const size_t o_hs = gimg_rb ? take((size_t)gimg_rb * 128 * d * 2) : off;
  if (out) {
    char *b = static_cast<char *>(base);
    out->counters = reinterpret_cast<int32_t *>(b + o_cnt);
    out->seg_cnt = reinterpret_cast<int32_t *>(b + o_segc);
    out->seg_off = reinterpret_cast<int32_t *>(b + o_sego);
    out->tok_idx = reinterpret_cast<int32_t *>(b + o_idx);
    out->tok_y = reinterpret_cast<int32_t *>(b + o_y);
    out->tok_c = reinterpret_cast<float *>(b + o_c);
    out->lse = reinterpret_cast<float *>(b + o_lse);
    out->zy = reinterpret_cast<float *>(b + o_zy);
    out->part = reinterpret_cast<float2 *>(b + o_part);
    out->seg_logp = reinterpret_cast<double *>(b + o_segl);
    out->ppo_c = reinterpret_cast<float *>(b + o_ppoc);
    out->ppo_L = reinterpret_cast<double *>(b + o_ppol);
    out->Hc = b + o_hc;
    out->bkt = reinterpret_cast<int32_t *>(b + o_bkt);
    out->blist = reinterpret_cast<int32_t *>(b + o_blist);
    out->gring = b + o_ring;
    out->tailbuf = cl ? reinterpret_cast<float *>(b + o_tail) : nullptr;
    out->ref = (cl || img) ? reinterpret_cast<float *>(b + o_ref) : nullptr;
    out->mrow = (cl || img) ? reinterpret_cast<float *>(b + o_mrow) : nullptr;
    out->lsum = img ? reinterpret_cast<float *>(b + o_lsum) : nullptr;
    out->prog = img ? reinterpret_cast<int32_t *>(b + o_prog) : nullptr;
    out->rbflag = cl ? reinterpret_cast<int32_t *>(b + o_rbflag) : nullptr;
    out->rb_list = cl ? reinterpret_cast<int32_t *>(b + o_rblist) : nullptr;
    out->ready = cl ? reinterpret_cast<int32_t *>(b + o_ready) : nullptr;
    out->lpart = cl ? reinterpret_cast<float *>(b + o_lpart) : nullptr;
    out->tail_l = cl ? reinterpret_cast<float *>(b + o_taill) : nullptr;
    out->n_rbmax = n_rbmax;
    out->n_slots = n_slots;
    out->gimg = gimg_rb ? b + o_gimg : nullptr;
    out->hs = gimg_rb ? b + o_hs : nullptr;
    out->gimg_rb = gimg_rb;
    out->Tpad = Tpad;
    out->nsplit = kNSplit;
  }
  return off;
}

int grad_gimg_rows_fit(int64_t T, int32_t d, int32_t V, int32_t R, pair_dtype dt,
                       size_t ws_bytes) {
  const size_t base = grad_workspace_bytes(T, d, V, R, dt, nullptr, nullptr, 0);
  if (ws_bytes < base) return -1;
  const int pref = grad_gimg_rows(T, d, V, dt);
  if (pref == 0) return 0;
  const size_t fit = (ws_bytes - base) / grad_image_block_bytes(d, V);
  return fit < (size_t)pref ? (int)fit : pref;
}

pair_status grad_prepare(const GradArgs &g, const GradWorkspace &w,
                         cudaStream_t s) {
  // Bucket counters of the one-hot dW part (bf16 path): counts, then the
  // offsets the scan writes, then the fill counters; cleared with one pass.
  const int nb = (g.V + kOneHotBucket - 1) / kOneHotBucket;
  const bool bf16 = g.dt == PAIR_BF16;
  PAIR_BEGIN("seg_count", s);
  seg_count_kernel<<<g.R, 256, 0, s>>>(g.R, (int)g.T, g.V, g.cu, g.mask, g.y, g.a, w.seg_cnt,
                                       w.counters, w.bkt, bf16 ? 3 * (nb + 1) : 0, g.dev_err);
  PAIR_LAUNCH_CHECK(s);
  const bool sum = g.R <= kGatherScanMax;
  if (!sum) {
    PAIR_BEGIN("seg_scan", s);
    seg_scan_kernel<<<1, 1024, 0, s>>>(g.R, w.seg_cnt, w.seg_off, w.counters);
    PAIR_LAUNCH_CHECK(s);
  }
  // Threads for the mean rollout (a block walks its rollout in steps of them).
  const int64_t mean = g.T / g.R;
  const int threads = mean > 512 ? 1024 : mean > 256 ? 512 : 256;
  PAIR_BEGIN("gather", s);
  gather_kernel<<<g.R, threads, 0, s>>>(g.R, (int)g.T, g.V, g.cu, g.mask, g.y, g.a, w.seg_cnt,
                                        sum, w.seg_off, w.counters, w.tok_idx, w.tok_y, w.tok_c,
                                        bf16 ? w.bkt : nullptr);
  PAIR_LAUNCH_CHECK(s);
  const size_t cu_smem = g.R + 1 <= kZeroCuSmem ? (size_t)(g.R + 1) * sizeof(int32_t) : 0;
  const int grid = (int)(ceil_div(g.T, 8) < 152 * 8 ? ceil_div(g.T, 8) : 152 * 8);
  PAIR_BEGIN("rows", s);
  if (bf16)
    rows_kernel<__nv_bfloat16><<<grid, 256, cu_smem, s>>>(
        g.T, w.Tpad, g.d, g.R, w.counters, w.tok_idx, w.tok_y,
        static_cast<const __nv_bfloat16 *>(g.H), static_cast<const __nv_bfloat16 *>(g.W),
        static_cast<__nv_bfloat16 *>(w.Hc), w.gimg_rb > 0 ? w.ref : nullptr, g.cu, g.mask, g.a,
        g.dH);
  else
    rows_kernel<float><<<grid, 256, cu_smem, s>>>(
        g.T, w.Tpad, g.d, g.R, w.counters, w.tok_idx, w.tok_y, static_cast<const float *>(g.H),
        static_cast<const float *>(g.W), static_cast<float *>(w.Hc), nullptr, g.cu, g.mask, g.a,
        g.dH);
  PAIR_LAUNCH_CHECK(s);
  return PAIR_OK;
}

pair_status grad_finalize(const GradArgs &g, const GradWorkspace &w,
                          cudaStream_t s) {
  PAIR_BEGIN("finalize", s);
  finalize_kernel<<<g.R, 256, 0, s>>>(g.R, w.seg_off, w.zy, w.lse, g.a, w.seg_logp, w.counters,
                                      g.Jobj, g.logp_seq);
  PAIR_LAUNCH_CHECK(s);
  return PAIR_OK;
}

pair_status grad_token_logp(int64_t T, const GradWorkspace &w, float *logp_tok,
                            cudaStream_t s) {
  PAIR_BEGIN("zero_logp", s);
  zero_f32_kernel<<<152 * 4, 256, 0, s>>>(T, logp_tok);
  PAIR_LAUNCH_CHECK(s);
  PAIR_BEGIN("scatter_logp", s);
  scatter_logp_kernel<<<152 * 4, 256, 0, s>>>(w.counters, w.tok_idx, w.zy, w.lse, logp_tok);
  PAIR_LAUNCH_CHECK(s);
  return PAIR_OK;
}

pair_status grad_ppo_coefficients(const GradArgs &g, const GradWorkspace &w,
                                  const float *logp_old, float eps, float *coef_out,
                                  cudaStream_t s) {
  PAIR_BEGIN("ppo_coef", s);
  ppo_coef_kernel<<<g.R, 256, 0, s>>>(g.R, w.seg_off, w.zy, w.lse, g.a, logp_old, eps,
                                      w.seg_logp, w.ppo_c, w.ppo_L, coef_out, w.tok_c);
  PAIR_LAUNCH_CHECK(s);
  return PAIR_OK;
}

pair_status grad_ppo_finalize(const GradArgs &g, const GradWorkspace &w, cudaStream_t s) {
  PAIR_BEGIN("ppo_objective", s);
  ppo_objective_kernel<<<1, 1024, 0, s>>>(g.R, g.a, w.seg_logp, w.ppo_L, g.Jobj, g.logp_seq);
  PAIR_LAUNCH_CHECK(s);
  return PAIR_OK;
}

pair_status grad_onehot(const GradArgs &g, const GradWorkspace &w,
                        cudaStream_t s) {
  const int nb = (g.V + kOneHotBucket - 1) / kOneHotBucket;
  int32_t *cnt = w.bkt, *off = w.bkt + (nb + 1), *fill = w.bkt + 2 * (nb + 1);
  PAIR_BEGIN("onehot_scan", s);
  onehot_scan_kernel<<<1, 1024, 0, s>>>(nb, cnt, off);
  PAIR_LAUNCH_CHECK(s);
  PAIR_BEGIN("onehot_fill", s);
  onehot_fill_kernel<<<152 * 4, 256, 0, s>>>(w.counters, w.tok_y, off, fill, w.blist);
  PAIR_LAUNCH_CHECK(s);
  const int blocks = (int)ceil_div(nb, 8);  // 8 warps (buckets) per block
  if (g.dt == PAIR_BF16) {
    const __nv_bfloat16 *W = static_cast<const __nv_bfloat16 *>(g.W);
    PAIR_BEGIN("onehot_dh", s);
    onehot_dh_kernel<__nv_bfloat16><<<152 * 16, 256, 0, s>>>(
        g.d, w.counters, w.tok_idx, w.tok_y, w.tok_c, W, g.dH);
    PAIR_LAUNCH_CHECK(s);
    PAIR_BEGIN("onehot_dw", s);
    onehot_dw_kernel<__nv_bfloat16><<<blocks, 256, 0, s>>>(
        g.d, g.V, nb, w.counters, w.tok_y, w.tok_c, off, w.blist,
        static_cast<const __nv_bfloat16 *>(w.Hc), g.dW);
    PAIR_LAUNCH_CHECK(s);
  } else {
    PAIR_BEGIN("onehot_dh", s);
    onehot_dh_kernel<float><<<152 * 16, 256, 0, s>>>(
        g.d, w.counters, w.tok_idx, w.tok_y, w.tok_c,
        static_cast<const float *>(g.W), g.dH);
    PAIR_LAUNCH_CHECK(s);
    PAIR_BEGIN("onehot_dw", s);
    onehot_dw_kernel<float><<<blocks, 256, 0, s>>>(
        g.d, g.V, nb, w.counters, w.tok_y, w.tok_c, off, w.blist,
        static_cast<const float *>(w.Hc), g.dW);
    PAIR_LAUNCH_CHECK(s);
  }
  return PAIR_OK;
}

}  // namespace pairk
