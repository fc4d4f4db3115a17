// fp32 LM-head path of pair_grad on the CUDA cores (PAIR_F32 inputs).
//
// The objective of Sec. 4.5, sum_i a_i log pi(o_i|q), over compacted active
// tokens t (coefficient c_t = a of its rollout):
//   z_tv = <h_t, W_v>, lse_t = log sum_v exp z_tv, logp_t = z_{t,y_t} - lse_t
//   dJ/dh_t = c_t W_{y_t} - c_t sum_v p_tv W_v,   p_tv = exp(z_tv - lse_t),
//   dJ/dW_v = sum_{t: y_t = v} c_t h_t - sum_t c_t p_tv h_t.
// Logits are recomputed where needed and never stored. Every reduction runs
// in a fixed order, so results are bit-reproducible. fp32 throughout; the
// one-hot terms are added last, so that the long sums only carry the softmax
// parts (about 1 / sqrt(V) of the whole).
#include <cooperative_groups.h>

#include "pair_common.cuh"

namespace pairk {
namespace {

namespace cg = cooperative_groups;

// ------------------------------------------------ tiled form, d <= 2048
//
// One kernel for both gradients, whose roles are symmetric: 32 rows of A
// (tokens for dH, vocabulary rows for dW) against 32-row tiles of B (the
// other side), and per tile
//     z = A B^T,   g = f(z),   out += g B,
// with B's tile read once from shared memory for both products. For dH the
// row's maximum and sum run along (out is rescaled when the maximum grows), so
// the log-sum-exp costs no pass of its own and the head takes four
// logit-sized products; for dW, g = -c_t exp(z - lse_t).
//
// 128 threads; 4 x 2 logits and 4 x 16 outputs a thread (6 and 5 shared-memory
// wavefronts for 8 and 16 cycles of multiply-adds), B double-buffered by
// cp.async, 108 KB, two CTAs per SM. A cluster is C x S CTAs: C slices of
// up to 256 columns of d, whose partial logits are added through distributed
// shared memory, and S parts of B, whose outputs are added at the end the same
// way, in rank order: 1075 tokens are 34 row tiles, too few for 304 CTA slots.
// What bounds it: fp32 multiply-adds (128 per clock and SM).
// Measured on one GB300, 4 x 8 rollouts of 32 to 64 tokens, d = 256, V = 4096:
// dH with the log-sum-exp 151 us (597 + 962 row by row, a block per token),
// dW 182 us (856): 30 and 25 TFLOP/s counting the recomputed logits.
constexpr int kBM = 32, kBN = 32, kTileThreads = 128;
constexpr int kSliceMax = 256;               // columns of d per CTA, at most
constexpr int kTileDMax = 8 * kSliceMax;     // largest d of this form
constexpr int kGPitch = kBM + 4;
enum { kModeLse = 0, kModeDh = 1, kModeDw = 2 };

struct TileArgs {
  int d, V, C, S;
  const int32_t *counters, *tok_idx, *tok_y;
  const float *tok_c, *Hc, *W;
  float *lse, *zy, *out;
};

__host__ __device__ __forceinline__ int tile_slice(int d, int C) {
  return ((d / 16 + C - 1) / C) * 16;
}
// 64-column groups of a slice: outputs per thread, and the pitch of a tile's
// rows (columns past the slice hold anything; their outputs are not used).
__host__ __device__ __forceinline__ int tile_groups(int slice) { return (slice + 63) / 64; }
inline size_t tile_smem(int d, int C) {
  const size_t pitch = tile_groups(tile_slice(d, C)) * 64 + 4;
  return sizeof(float) * ((kBM + 2 * kBN) * pitch   // A, B (two buffers)
                          + kBN * kGPitch           // g, n-major
                          + 2 * kBM * kBN           // partial logits (two buffers)
                          + 4 * kBM);               // row maximum, sum, rescaling, target logit
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// 32 rows [r0, r0 + 32) x columns [k0, k0 + n) of src [rows][d] into dst
// (pitch floats per row); rows past the end are zero.
__device__ __forceinline__ void load_tile(float *dst, int pitch, const float *src, int rows,
                                          int r0, int d, int k0, int n) {
  const int n4 = n / 4;
  for (int e = threadIdx.x; e < 32 * n4; e += kTileThreads) {
    const int i = e / n4, k = (e - i * n4) * 4;
    float *q = dst + i * pitch + k;
    if (r0 + i < rows) cp_async16(q, src + (size_t)(r0 + i) * d + k0 + k);
    else *reinterpret_cast<float4 *>(q) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

template <int MODE, int NJ>
__global__ void __launch_bounds__(kTileThreads, 2) simt_tile_kernel(const TileArgs g) {
  const int Teff = g.counters[0];
  const int C = g.C, S = g.S, cs = C * S;
  const int m0 = (int)(blockIdx.x / cs) * kBM;
  const int M = MODE == kModeDw ? g.V : Teff, N = MODE == kModeDw ? Teff : g.V;
  if (m0 >= M) return;  // the whole cluster
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), ci = rank % C, si = rank / C;
  const int d = g.d, ds = tile_slice(d, C), k0 = ci * ds;
  const int dn = max(min(ds, d - k0), 0);  // this CTA's columns (a multiple of 16)
  constexpr int pitch = NJ * 64 + 4;
  const float *A = MODE == kModeDw ? g.W : g.Hc, *B = MODE == kModeDw ? g.Hc : g.W;

  extern __shared__ __align__(16) float smem[];
  float *As = smem, *Bs = As + kBM * pitch, *Gs = Bs + 2 * kBN * pitch;
  float *Zp = Gs + kBN * kGPitch, *rm = Zp + 2 * kBM * kBN, *rl = rm + kBM, *rf = rl + kBM, *rz = rf + kBM;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // Logits: rows zm * 4 + i, columns zn + 16 j. Outputs: rows om * 4 + i,
  // columns oc * 4 + 64 j.
  const int zm = (warp & 1) * 4 + lane / 8, zn = (warp >> 1) * 8 + lane % 8;
  const int om = zm, oc = zn;

  // Tiles of this part of B; every CTA of the cluster runs the same number
  // of steps (they exchange partial logits in each).
  const int nt = (N + kBN - 1) / kBN;
  const int t0 = (int)((int64_t)si * nt / S), t1 = (int)((int64_t)(si + 1) * nt / S);
  const int steps = (nt + S - 1) / S;

  if (tid < kBM) {
    rm[tid] = -INFINITY;
    rl[tid] = 0.f;
    rz[tid] = 0.f;  // the part that holds the target's tile sets it
  }
  // The target of softmax row tid / 4.
  const int ytile =
      MODE != kModeDw && m0 + tid / 4 < Teff ? g.tok_y[m0 + tid / 4] : -1;
  float acc[4][NJ][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;

  load_tile(As, pitch, A, M, m0, d, k0, dn);
  if (t0 < t1) load_tile(Bs, pitch, B, N, t0 * kBN, d, k0, dn);
  cp_async_commit();

  for (int st = 0; st < steps; ++st) {
    const int t = t0 + st, n0 = t * kBN;
    const bool live = t < t1;
    const float *Bt = Bs + (st & 1) * kBN * pitch;
    cp_async_wait<0>();
    __syncthreads();  // this tile is in; the other buffer and Gs are free
    if (t + 1 < t1) load_tile(Bs + ((st + 1) & 1) * kBN * pitch, pitch, B, N, n0 + kBN, d, k0, dn);
    cp_async_commit();

    float z[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i][0] = z[i][1] = 0.f;
    if (live) {
      // 16-column pieces summed apart (shorter chains of roundings); the
      // operands of the next 4 columns are loaded while these are multiplied.
      const float *ap = As + zm * 4 * pitch, *bp = Bt + zn * pitch;
      float4 a[2][4], b[2][2];
      auto fetch = [&](int k, int q) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          a[q][i] = *reinterpret_cast<const float4 *>(ap + i * pitch + k);
#pragma unroll
        for (int j = 0; j < 2; ++j)
          b[q][j] = *reinterpret_cast<const float4 *>(bp + 16 * j * pitch + k);
      };
      fetch(0, 0);
      for (int k = 0; k < dn; k += 16) {
        float zc[4][2];
#pragma unroll
        for (int i = 0; i < 4; ++i) zc[i][0] = zc[i][1] = 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          // (Past the slice's end: still inside the row's pitch.)
          fetch(k + 4 * u + 4, (u + 1) & 1);
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              zc[i][j] = fmaf(a[u & 1][i].x, b[u & 1][j].x, zc[i][j]);
              zc[i][j] = fmaf(a[u & 1][i].y, b[u & 1][j].y, zc[i][j]);
              zc[i][j] = fmaf(a[u & 1][i].z, b[u & 1][j].z, zc[i][j]);
              zc[i][j] = fmaf(a[u & 1][i].w, b[u & 1][j].w, zc[i][j]);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j) z[i][j] += zc[i][j];
      }
    }
    if (C > 1) {
      float *zp = Zp + (st & 1) * kBM * kBN;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) zp[(zm * 4 + i) * kBN + zn + 16 * j] = z[i][j];
      cluster.sync();
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) z[i][j] = 0.f;
      for (int c = 0; c < C; ++c) {
        const float *q = cluster.map_shared_rank(zp, si * C + c);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j) z[i][j] += q[(zm * 4 + i) * kBN + zn + 16 * j];
      }
    }
    if (!live) continue;  // uniform over the CTA

    bool rescale = false;
    if constexpr (MODE == kModeDw) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int n = n0 + zn + 16 * j;
        const bool in = n < N;
        const float c = in ? g.tok_c[n] : 0.f, ls = in ? g.lse[n] : 0.f;
        float v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = in ? -c * expf(z[i][j] - ls) : 0.f;
        *reinterpret_cast<float4 *>(Gs + (zn + 16 * j) * kGPitch + zm * 4) =
            make_float4(v[0], v[1], v[2], v[3]);
      }
      __syncthreads();
    } else {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const bool in = n0 + zn + 16 * j < N;
        *reinterpret_cast<float4 *>(Gs + (zn + 16 * j) * kGPitch + zm * 4) =
            in ? make_float4(z[0][j], z[1][j], z[2][j], z[3][j])
               : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      }
      __syncthreads();
      // Row m = tid / 4: four lanes, eight columns each.
      const int m = tid / 4, q = tid & 3;
      float v[8], mx = -INFINITY;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        v[u] = Gs[(4 * u + q) * kGPitch + m];
        mx = fmaxf(mx, v[u]);
        if (n0 + 4 * u + q == ytile) rz[m] = v[u];
      }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float old = rm[m], now = fmaxf(old, mx);
      float l = 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        v[u] = expf(v[u] - now);
        l += v[u];
        if (MODE == kModeDh) Gs[(4 * u + q) * kGPitch + m] = v[u];
      }
      l += __shfl_xor_sync(0xffffffffu, l, 1);
      l += __shfl_xor_sync(0xffffffffu, l, 2);
      const float f = expf(old - now);  // 0 at the first tile
      if (q == 0) {
        rl[m] = fmaf(rl[m], f, l);
        rm[m] = now;
        rf[m] = f;
      }
      rescale = __syncthreads_or(f != 1.f);
    }
    if constexpr (MODE != kModeLse) {
      if (rescale) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float f = rf[om * 4 + i];
#pragma unroll
          for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] *= f;
        }
      }
      const float *gp = Gs + om * 4, *bp = Bt + oc * 4;
      float4 gv = *reinterpret_cast<const float4 *>(gp), b[NJ];
#pragma unroll
      for (int j = 0; j < NJ; ++j) b[j] = *reinterpret_cast<const float4 *>(bp + 64 * j);
#pragma unroll 4
      for (int n = 0; n < kBN; ++n) {
        const float gi[4] = {gv.x, gv.y, gv.z, gv.w};
        float4 c[NJ];
#pragma unroll
        for (int j = 0; j < NJ; ++j) c[j] = b[j];
        const int nn = n + 1 < kBN ? n + 1 : n;  // the next row, while this one is multiplied
        gv = *reinterpret_cast<const float4 *>(gp + nn * kGPitch);
#pragma unroll
        for (int j = 0; j < NJ; ++j)
          b[j] = *reinterpret_cast<const float4 *>(bp + nn * pitch + 64 * j);
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            acc[i][j][0] = fmaf(gi[i], c[j].x, acc[i][j][0]);
            acc[i][j][1] = fmaf(gi[i], c[j].y, acc[i][j][1]);
            acc[i][j][2] = fmaf(gi[i], c[j].z, acc[i][j][2]);
            acc[i][j][3] = fmaf(gi[i], c[j].w, acc[i][j][3]);
          }
      }
    }
  }

  // ---- the parts' results, added in rank order. This CTA writes rows
  // [r0, r1) of the tile, its own columns.
  cp_async_wait<0>();  // (A's rows, where there was no tile to wait for)
  __syncthreads();
  float *Os = Bs;  // [32][pitch]
  if constexpr (MODE != kModeLse) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        *reinterpret_cast<float4 *>(Os + (om * 4 + i) * pitch + oc * 4 + 64 * j) =
            make_float4(acc[i][j][0], acc[i][j][1], acc[i][j][2], acc[i][j][3]);
  }
  cluster.sync();
  const int r0 = si * kBM / S, r1 = (si + 1) * kBM / S;
  if constexpr (MODE != kModeDw) {
    // Maximum and sum of each row over the parts, one row per warp at a time.
    for (int r = r0 + warp; r < r1; r += kTileThreads / 32) {
      const int p = m0 + r;
      if (p >= Teff) break;
      float Mx = -INFINITY, L = 0.f;
      for (int s = 0; s < S; ++s) Mx = fmaxf(Mx, cluster.map_shared_rank(rm, s * C + ci)[r]);
      for (int s = 0; s < S; ++s) {
        const float ms = cluster.map_shared_rank(rm, s * C + ci)[r];
        if (ms > -INFINITY) L += cluster.map_shared_rank(rl, s * C + ci)[r] * expf(ms - Mx);
      }
      const int y = g.tok_y[p];
      if (ci == 0 && lane == 0) {
        float zt = 0.f;
        for (int s = 0; s < S; ++s) zt += cluster.map_shared_rank(rz, s * C + ci)[r];
        g.lse[p] = Mx + logf(L);
        g.zy[p] = zt;
      }
      if constexpr (MODE == kModeDh) {
        const float c = g.tok_c[p], sc = c != 0.f ? -c / L : 0.f;
        float *row = g.out + (size_t)g.tok_idx[p] * d + k0;
        for (int k = lane * 4; k < dn; k += 128) {
          float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int s = 0; s < S; ++s) {
            const float ms = cluster.map_shared_rank(rm, s * C + ci)[r];
            if (!(ms > -INFINITY)) continue;
            const float f = expf(ms - Mx);
            const float4 v = *reinterpret_cast<const float4 *>(
                cluster.map_shared_rank(Os, s * C + ci) + r * pitch + k);
            o.x = fmaf(f, v.x, o.x); o.y = fmaf(f, v.y, o.y);
            o.z = fmaf(f, v.z, o.z); o.w = fmaf(f, v.w, o.w);
          }
          const float4 w = *reinterpret_cast<const float4 *>(g.W + (size_t)y * d + k0 + k);
          *reinterpret_cast<float4 *>(row + k) =
              make_float4(fmaf(c, w.x, sc * o.x), fmaf(c, w.y, sc * o.y), fmaf(c, w.z, sc * o.z),
                          fmaf(c, w.w, sc * o.w));
        }
      }
    }
  } else {
    // Rows into As (free by now), the one-hot terms of their tokens in
    // packed order on top, then out. Each thread keeps to its columns.
    for (int r = r0; r < r1; ++r)
      for (int k = tid * 4; k < dn; k += kTileThreads * 4) {
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s = 0; s < S; ++s) {
          const float4 v = *reinterpret_cast<const float4 *>(
              cluster.map_shared_rank(Os, s * C + ci) + r * pitch + k);
          o.x += v.x; o.y += v.y; o.z += v.z; o.w += v.w;
        }
        *reinterpret_cast<float4 *>(As + r * pitch + k) = o;
      }
    const int v0 = m0 + r0, v1 = min(m0 + r1, g.V);
    for (int p0 = 0; p0 < Teff; p0 += 32) {
      // Every warp finds the same hits.
      const int y = p0 + lane < Teff ? g.tok_y[p0 + lane] : -1;
      unsigned hit = __ballot_sync(0xffffffffu, y >= v0 && y < v1);
      while (hit) {
        const int src = __ffs(hit) - 1;
        hit &= hit - 1;
        const int r = __shfl_sync(0xffffffffu, y, src) - m0, p = p0 + src;
        const float c = g.tok_c[p];
        for (int k = tid * 4; k < dn; k += kTileThreads * 4) {
          const float4 h = *reinterpret_cast<const float4 *>(g.Hc + (size_t)p * d + k0 + k);
          float4 *o = reinterpret_cast<float4 *>(As + r * pitch + k);
          *o = make_float4(fmaf(c, h.x, o->x), fmaf(c, h.y, o->y), fmaf(c, h.z, o->z),
                           fmaf(c, h.w, o->w));
        }
      }
    }
    for (int r = r0; r < r1; ++r)
      if (m0 + r < g.V)
        for (int k = tid * 4; k < dn; k += kTileThreads * 4)
          *reinterpret_cast<float4 *>(g.out + (size_t)(m0 + r) * d + k0 + k) =
              *reinterpret_cast<const float4 *>(As + r * pitch + k);
  }
  cluster.sync();  // the peers' shared memory stays up while it is read
}

template <int MODE, int NJ>
pair_status launch_tile_nj(const char *name, const TileArgs &a, int64_t ctas, size_t smem,
                           cudaStream_t s) {
  PAIR_CUDA_TRY(cudaFuncSetAttribute(simt_tile_kernel<MODE, NJ>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ctas, 1, 1);
  cfg.blockDim = dim3(kTileThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = a.C * a.S;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  PAIR_BEGIN(name, s);
  PAIR_CUDA_TRY(cudaLaunchKernelEx(&cfg, simt_tile_kernel<MODE, NJ>, a));
  PAIR_LAUNCH_CHECK(s);
  return PAIR_OK;
}

template <int MODE>
pair_status launch_tile(const char *name, const GradArgs &g, const GradWorkspace &w, float *out,
                        cudaStream_t s) {
  // Row and column counts as far as the host knows them (T for tokens).
  const int64_t M = MODE == kModeDw ? g.V : g.T, N = MODE == kModeDw ? g.T : g.V;
  int C = 1;
  while (tile_slice(g.d, C) > kSliceMax) C *= 2;
  // Parts of B: enough CTAs for two on each of the 152 SMs (of T packed
  // tokens fewer are active, so rounded up), at least one tile each.
  const int64_t tiles = ceil_div(M, kBM);
  int S = 1;
  while (S * C < 8 && tiles * C * S < 304 && 2 * S <= ceil_div(N, kBN)) S *= 2;
  const size_t smem = tile_smem(g.d, C);
  const TileArgs a{g.d, g.V, C, S, w.counters, w.tok_idx, w.tok_y, w.tok_c,
                   static_cast<const float *>(w.Hc), static_cast<const float *>(g.W),
                   w.lse, w.zy, out};
  const int64_t ctas = tiles * C * S;
  switch (tile_groups(tile_slice(g.d, C))) {
    case 1: return launch_tile_nj<MODE, 1>(name, a, ctas, smem, s);
    case 2: return launch_tile_nj<MODE, 2>(name, a, ctas, smem, s);
    case 3: return launch_tile_nj<MODE, 3>(name, a, ctas, smem, s);
    default: return launch_tile_nj<MODE, 4>(name, a, ctas, smem, s);
  }
}

// ------------------------------------------------ any d (above 2048)

constexpr int kWarps = 8;

__device__ __forceinline__ float warp_sum(float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// lse and target logit of every active token: one block per token, one warp
// per vocabulary row (coalesced W reads), online max / sum-exp per warp.
__global__ void __launch_bounds__(kWarps * 32) simt_lse_kernel(
    int d, int V, const int32_t *counters, const float *Hc, const float *W,
    const int32_t *tok_y, float *lse, float *zy) {
  extern __shared__ float hs[];
  __shared__ float wm[kWarps], wl[kWarps], wz[kWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Teff = counters[0];
  for (int p = blockIdx.x; p < Teff; p += gridDim.x) {
    for (int k = threadIdx.x; k < d; k += blockDim.x) hs[k] = Hc[(int64_t)p * d + k];
    __syncthreads();
    const int yt = tok_y[p];
    float m = -INFINITY, l = 0.f, zt = 0.f;
    for (int v = warp; v < V; v += kWarps) {
      const float *w = W + (int64_t)v * d;
      float z = 0.f;
      for (int k = lane; k < d; k += 32) z = fmaf(hs[k], w[k], z);
      z = warp_sum(z);
      const float mn = fmaxf(m, z);
      l = l * expf(m - mn) + expf(z - mn);
      m = mn;
      if (v == yt) zt = z;
    }
    if (lane == 0) { wm[warp] = m; wl[warp] = l; wz[warp] = zt; }
    __syncthreads();
    if (threadIdx.x == 0) {
      float M = -INFINITY;
      for (int k = 0; k < kWarps; ++k) M = fmaxf(M, wm[k]);
      float L = 0.f, Z = 0.f;
      for (int k = 0; k < kWarps; ++k) {
        L += wl[k] * expf(wm[k] - M);
        if ((yt % kWarps) == k) Z = wz[k];
      }
      lse[p] = M + logf(L);
      zy[p] = Z;
    }
    __syncthreads();
  }
}

// dJ/dh_t for every active token: one block per token; warp w accumulates
// vocabulary rows v = w mod kWarps into its own shared-memory row.
__global__ void __launch_bounds__(kWarps * 32) simt_dh_kernel(
    int d, int V, const int32_t *counters, const int32_t *tok_idx,
    const float *Hc, const float *W, const int32_t *tok_y, const float *tok_c,
    const float *lse, float *dH) {
  extern __shared__ float sm[];
  float *hs = sm;            // [d]
  float *acc = sm + d;       // [kWarps][d]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Teff = counters[0];
  for (int p = blockIdx.x; p < Teff; p += gridDim.x) {
    for (int k = threadIdx.x; k < d; k += blockDim.x) hs[k] = Hc[(int64_t)p * d + k];
    for (int k = threadIdx.x; k < kWarps * d; k += blockDim.x) acc[k] = 0.f;
    __syncthreads();
    const int yt = tok_y[p];
    const float c = tok_c[p], ls = lse[p];
    float *my = acc + warp * d;
    for (int v = warp; v < V; v += kWarps) {
      const float *w = W + (int64_t)v * d;
      float z = 0.f;
      for (int k = lane; k < d; k += 32) z = fmaf(hs[k], w[k], z);
      z = warp_sum(z);
      const float g = c * ((v == yt ? 1.f : 0.f) - expf(z - ls));
      for (int k = lane; k < d; k += 32) my[k] = fmaf(g, w[k], my[k]);
    }
    __syncthreads();
    float *row = dH + (int64_t)tok_idx[p] * d;
    for (int k = threadIdx.x; k < d; k += blockDim.x) {
      float s = 0.f;
      for (int q = 0; q < kWarps; ++q) s += acc[q * d + k];
      row[k] = s;
    }
    __syncthreads();
  }
}

// dJ/dW_v for every vocabulary row: one block per row; warp w accumulates
// active tokens p = w mod kWarps.
__global__ void __launch_bounds__(kWarps * 32) simt_dw_kernel(
    int d, int V, const int32_t *counters, const float *Hc, const float *W,
    const int32_t *tok_y, const float *tok_c, const float *lse, float *dW) {
  extern __shared__ float sm[];
  float *ws = sm;            // [d]
  float *acc = sm + d;       // [kWarps][d]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Teff = counters[0];
  for (int v = blockIdx.x; v < V; v += gridDim.x) {
    for (int k = threadIdx.x; k < d; k += blockDim.x) ws[k] = W[(int64_t)v * d + k];
    for (int k = threadIdx.x; k < kWarps * d; k += blockDim.x) acc[k] = 0.f;
    __syncthreads();
    float *my = acc + warp * d;
    for (int p = warp; p < Teff; p += kWarps) {
      const float *h = Hc + (int64_t)p * d;
      float z = 0.f;
      for (int k = lane; k < d; k += 32) z = fmaf(ws[k], h[k], z);
      z = warp_sum(z);
      const float g = tok_c[p] * ((tok_y[p] == v ? 1.f : 0.f) - expf(z - lse[p]));
      for (int k = lane; k < d; k += 32) my[k] = fmaf(g, h[k], my[k]);
    }
    __syncthreads();
    float *row = dW + (int64_t)v * d;
    for (int k = threadIdx.x; k < d; k += blockDim.x) {
      float s = 0.f;
      for (int q = 0; q < kWarps; ++q) s += acc[q * d + k];
      row[k] = s;
    }
    __syncthreads();
  }
}

}  // namespace

pair_status grad_lse_simt(const GradArgs &g, const GradWorkspace &w, cudaStream_t s) {
  if (g.d <= kTileDMax) return launch_tile<kModeLse>("simt_lse", g, w, nullptr, s);
  const float *Hc = static_cast<const float *>(w.Hc);
  const float *W = static_cast<const float *>(g.W);
  const int grid = 152 * 8;
  const size_t sm1 = (size_t)g.d * 4;
  PAIR_CUDA_TRY(cudaFuncSetAttribute(simt_lse_kernel,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm1));
  PAIR_BEGIN("simt_lse", s);
  simt_lse_kernel<<<grid, kWarps * 32, sm1, s>>>(g.d, g.V, w.counters, Hc, W, w.tok_y, w.lse,
                                                 w.zy);
  PAIR_LAUNCH_CHECK(s);
  return PAIR_OK;
}

pair_status grad_bwd_simt(const GradArgs &g, const GradWorkspace &w, cudaStream_t s) {
  if (g.d <= kTileDMax) {
    // dH with its log-sum-exp (the same values again after grad_lse_simt).
    const pair_status st = launch_tile<kModeDh>("simt_dh", g, w, g.dH, s);
    return st != PAIR_OK ? st : launch_tile<kModeDw>("simt_dw", g, w, g.dW, s);
  }
  const float *Hc = static_cast<const float *>(w.Hc);
  const float *W = static_cast<const float *>(g.W);
  const int grid = 152 * 8;
  const size_t sm2 = (size_t)(kWarps + 1) * g.d * 4;
  PAIR_CUDA_TRY(cudaFuncSetAttribute(simt_dh_kernel,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm2));
  PAIR_CUDA_TRY(cudaFuncSetAttribute(simt_dw_kernel,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm2));
  PAIR_BEGIN("simt_dh", s);
  simt_dh_kernel<<<grid, kWarps * 32, sm2, s>>>(g.d, g.V, w.counters, w.tok_idx, Hc, W, w.tok_y,
                                                w.tok_c, w.lse, g.dH);
  PAIR_LAUNCH_CHECK(s);
  const int gridv = (int)(g.V < 152 * 16 ? g.V : 152 * 16);
  PAIR_BEGIN("simt_dw", s);
  simt_dw_kernel<<<gridv, kWarps * 32, sm2, s>>>(g.d, g.V, w.counters, Hc, W, w.tok_y, w.tok_c,
                                                 w.lse, g.dW);
  PAIR_LAUNCH_CHECK(s);
  return PAIR_OK;
}

pair_status grad_head_simt(const GradArgs &g, const GradWorkspace &w, cudaStream_t s) {
  if (g.d <= kTileDMax) return grad_bwd_simt(g, w, s);
  const pair_status st = grad_lse_simt(g, w, s);
  return st != PAIR_OK ? st : grad_bwd_simt(g, w, s);
}

}  // namespace pairk
