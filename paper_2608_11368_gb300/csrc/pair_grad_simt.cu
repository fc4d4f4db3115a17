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
// 128 threads, two CTAs per SM (three up to 128 columns). What bounds it is the
// latency between dependent steps with eight warps on an SM: the FMA pipe is
// busy 50 % of the cycles and shared memory's data path 48 %, and most of the
// rest are instructions that wait a fixed time for the one before. So a step does
// much with little: two multiply-adds an instruction, and thread tiles as large
// as the registers allow. Logits: each warp takes a quarter of the columns of d
// and all 32 x 32 of them, 8 x 4 a thread (12 16-byte loads for 128
// multiply-adds; 4 x 2 a thread over all columns took 24), and the four partial
// sums meet in shared memory. Outputs: 8 rows x 8 columns a thread. A cluster is
// C x S CTAs: C slices of up to 256 columns of d, whose partial logits are added
// through distributed shared memory, and S parts of B, whose outputs are added
// at the end the same way, in rank order: 1075 tokens are 34 row tiles, too few
// for 304 CTA slots. 1,075 active tokens, d = 256, V = 4,096: dH with its
// log-sum-exp 133 us, dW 145 us (single multiply-adds on smaller thread tiles:
// 166 and 192 us); the four products are 9.0 GFLOP, 0.12 ms at the FMA rate.
constexpr int kBM = 32, kBN = 32, kTileThreads = 128;
constexpr int kSliceMax = 256;               // columns of d per CTA, at most
constexpr int kTileDMax = 8 * kSliceMax;     // largest d of this form
constexpr int kGPitch = kBM + 8;   // g, n-major: writes of a row's columns miss each other
constexpr int kZPitch = kBN + 4;   // partial logits of a warp
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
// 128-column groups of a slice: outputs per thread, and the pitch of a tile's
// rows (columns past the slice hold anything; their outputs are not used).
__host__ __device__ __forceinline__ int tile_groups(int slice) { return (slice + 127) / 128; }
inline size_t tile_smem(int d, int C) {
  const size_t pitch = tile_groups(tile_slice(d, C)) * 128 + 4;
  return sizeof(float) * ((kBM + kBN) * pitch            // A, B
                          + kBN * kGPitch                // g, n-major
                          + 4 * kBM * kZPitch            // the warps' partial logits
                          + (C > 1 ? 2 * kBM * kBN : 0)  // the slices' (two buffers)
                          + 4 * kBM                      // row maximum, sum, rescaling, target logit
                          + 2 * kBN);                    // dW: lse and -c of the tile's tokens
}

// Two fp32 multiply-adds in one instruction (each rounded like fmaf): half the
// issue slots of the products' inner loops.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<unsigned long long &>(d))
      : "l"(reinterpret_cast<unsigned long long &>(a)),
        "l"(reinterpret_cast<unsigned long long &>(b)),
        "l"(reinterpret_cast<unsigned long long &>(c)));
  return d;
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
__global__ void __launch_bounds__(kTileThreads, NJ == 1 ? 3 : 2)
    simt_tile_kernel(const TileArgs g) {
  const int Teff = g.counters[0];
  const int C = g.C, S = g.S, cs = C * S;
  const int m0 = (int)(blockIdx.x / cs) * kBM;
  const int M = MODE == kModeDw ? g.V : Teff, N = MODE == kModeDw ? Teff : g.V;
  if (m0 >= M) return;  // the whole cluster
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), ci = rank % C, si = rank / C;
  const int d = g.d, ds = tile_slice(d, C), k0 = ci * ds;
  const int dn = max(min(ds, d - k0), 0);  // this CTA's columns (a multiple of 16)
  constexpr int pitch = NJ * 128 + 4;
  const float *A = MODE == kModeDw ? g.W : g.Hc, *B = MODE == kModeDw ? g.Hc : g.W;

  extern __shared__ __align__(16) float smem[];
  float *As = smem, *Bs = As + kBM * pitch, *Gs = Bs + kBN * pitch;
  float *Zw = Gs + kBN * kGPitch, *Zp = Zw + 4 * kBM * kZPitch;
  float *rm = Zp + (C > 1 ? 2 * kBM * kBN : 0), *rl = rm + kBM, *rf = rl + kBM, *rz = rf + kBM;
  float *tl = rz + kBM, *tc = tl + kBN;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // Partial logits: rows zm + 4 i, columns zn + 8 j (neighbouring rows: the
  // lanes of a load miss each other's banks). Summed logits and their softmax:
  // row m, columns 4 u + q. Outputs: rows warp * 8 + i, columns lane * 4 + 128 j.
  const int zm = lane / 8, zn = lane % 8, m = tid / 4, q = tid & 3;

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
  const int ytile = MODE != kModeDw && m0 + m < Teff ? g.tok_y[m0 + m] : -1;
  float2 acc[8][NJ][2];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[i][j][0] = acc[i][j][1] = make_float2(0.f, 0.f);

  load_tile(As, pitch, A, M, m0, d, k0, dn);
  if (t0 < t1) load_tile(Bs, pitch, B, N, t0 * kBN, d, k0, dn);
  cp_async_commit();

  for (int st = 0; st < steps; ++st) {
    const int t = t0 + st, n0 = t * kBN;
    const bool live = t < t1;
    if (st > 0) {
      __syncthreads();  // the tile before, Gs and Zw are free
      if (live) load_tile(Bs, pitch, B, N, n0, d, k0, dn);
      cp_async_commit();
    }
    if (MODE == kModeDw && tid < kBN && live) {
      const bool in = n0 + tid < N;
      tl[tid] = in ? g.lse[n0 + tid] : 0.f;
      tc[tid] = in ? -g.tok_c[n0 + tid] : 0.f;
    }
    cp_async_wait<0>();
    __syncthreads();  // this tile is in

    float z[8];
    if (live) {
      // This warp's 16-column pieces; even and odd columns summed apart.
      float2 zc[8][4];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) zc[i][j] = make_float2(0.f, 0.f);
      const float *ap = As + zm * pitch, *bp = Bs + zn * pitch;
      for (int k = warp * 16; k < dn; k += 64) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float4 a[8], b[4];
#pragma unroll
          for (int i = 0; i < 8; ++i)
            a[i] = *reinterpret_cast<const float4 *>(ap + 4 * i * pitch + k + 4 * u);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            b[j] = *reinterpret_cast<const float4 *>(bp + 8 * j * pitch + k + 4 * u);
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
              zc[i][j] = fma2(make_float2(a[i].x, a[i].y), make_float2(b[j].x, b[j].y), zc[i][j]);
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
              zc[i][j] = fma2(make_float2(a[i].z, a[i].w), make_float2(b[j].z, b[j].w), zc[i][j]);
        }
      }
      float *zw = Zw + warp * kBM * kZPitch;
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          zw[(zm + 4 * i) * kZPitch + zn + 8 * j] = zc[i][j].x + zc[i][j].y;
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float *p = Zw + m * kZPitch + 4 * u + q;
        constexpr int w = kBM * kZPitch;
        z[u] = (p[0] + p[w]) + (p[2 * w] + p[3 * w]);
      }
    }
    if (C > 1) {
      float *zp = Zp + (st & 1) * kBM * kBN;
      if (live)
#pragma unroll
        for (int u = 0; u < 8; ++u) zp[u * kTileThreads + tid] = z[u];
      cluster.sync();
      if (live) {
#pragma unroll
        for (int u = 0; u < 8; ++u) z[u] = 0.f;
        for (int c = 0; c < C; ++c) {
          const float *p = cluster.map_shared_rank(zp, si * C + c);
#pragma unroll
          for (int u = 0; u < 8; ++u) z[u] += p[u * kTileThreads + tid];
        }
      }
    }
    if (!live) continue;  // uniform over the CTA

    bool rescale = false;
    if constexpr (MODE == kModeDw) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int n = 4 * u + q;
        Gs[n * kGPitch + m] = n0 + n < N ? tc[n] * expf(z[u] - tl[n]) : 0.f;
      }
      __syncthreads();
    } else {
      // Four lanes per row, eight columns each.
      float mx = -INFINITY;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (n0 + 4 * u + q >= N) z[u] = -INFINITY;
        mx = fmaxf(mx, z[u]);
        if (n0 + 4 * u + q == ytile) rz[m] = z[u];
      }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float old = rm[m], now = fmaxf(old, mx);
      float l = 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        z[u] = expf(z[u] - now);
        l += z[u];
        if (MODE == kModeDh) Gs[(4 * u + q) * kGPitch + m] = z[u];
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
        for (int i = 0; i < 8; ++i) {
          const float f = rf[warp * 8 + i];
#pragma unroll
          for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              acc[i][j][e].x *= f;
              acc[i][j][e].y *= f;
            }
        }
      }
      const float *gp = Gs + warp * 8, *bp = Bs + lane * 4;
#pragma unroll 4
      for (int n = 0; n < kBN; ++n) {
        const float4 g0 = *reinterpret_cast<const float4 *>(gp + n * kGPitch);
        const float4 g1 = *reinterpret_cast<const float4 *>(gp + n * kGPitch + 4);
        const float gi[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          const float4 b = *reinterpret_cast<const float4 *>(bp + n * pitch + 128 * j);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float2 gg = make_float2(gi[i], gi[i]);
            acc[i][j][0] = fma2(gg, make_float2(b.x, b.y), acc[i][j][0]);
            acc[i][j][1] = fma2(gg, make_float2(b.z, b.w), acc[i][j][1]);
          }
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
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        *reinterpret_cast<float4 *>(Os + (warp * 8 + i) * pitch + lane * 4 + 128 * j) =
            make_float4(acc[i][j][0].x, acc[i][j][0].y, acc[i][j][1].x, acc[i][j][1].y);
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
  const int nj = tile_groups(tile_slice(g.d, C));
  // Parts of B, at least one tile each: doubled until the CTAs fill the 152 SMs,
  // which for dW, whose rows are all there, four fifths of the slots do (V =
  // 4,096, d = 256: 145 us in 256 CTAs, 162 in 512; 3,000: 65 us in 376, 76 in
  // 188) and a few more than all of them don't (V = 5,000, d = 512: 231 us in
  // 314 CTAs, 194 in 628). Of T packed tokens about two thirds are active, so
  // for dH all slots are wanted.
  const int64_t tiles = ceil_div(M, kBM), slots = 152 * (nj == 1 ? 3 : 2);
  const auto wants = [&](int64_t ctas) {
    if (MODE != kModeDw) return ctas < slots;
    return 5 * ctas < 4 * slots || (ctas > slots && 10 * ctas < 11 * slots);
  };
  int S = 1;
  while (S * C < 8 && 2 * S <= ceil_div(N, kBN) && wants(tiles * C * S)) S *= 2;
  const size_t smem = tile_smem(g.d, C);
  const TileArgs a{g.d, g.V, C, S, w.counters, w.tok_idx, w.tok_y, w.tok_c,
                   static_cast<const float *>(w.Hc), static_cast<const float *>(g.W),
                   w.lse, w.zy, out};
  const int64_t ctas = tiles * C * S;
  return nj == 1 ? launch_tile_nj<MODE, 1>(name, a, ctas, smem, s)
                                              : launch_tile_nj<MODE, 2>(name, a, ctas, smem, s);
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
