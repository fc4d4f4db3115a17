// pair_audit: the frozen-population estimator audit (Sec. 5, "Frozen-policy
// estimator audit"; App. D metrics) over many design draws of one candidate
// group with explicit score vectors s_i in R^D.
//
// Target: the complete-pair gradient g = scale * sum_{i<j} h_ij over all G
// candidates (Eq. pair-kernel), i.e. g = sum_i abar_i s_i with
// abar_i = scale * 1/2 sum_{j != i} (r_i - r_j). Every draw's estimate is
// ghat_b = sum_i a_bi s_i (the coefficient collapse of Eq. pair-ht, under any
// weighting of pair_coeffs_weighted), so with the Gram matrix K = S S^T all
// statistics are G-dimensional quadratic forms:
//   ||ghat_b - g||^2 = e_b^T K e_b,  e_b = a_b - abar,
//   <ghat_b, g> = a_b^T K abar,  ||ghat_b||^2 = a_b^T K a_b,
//   E[ghat] - g = (E[a] - abar) S.
// K, abar, the coefficients' division, centring and scale and the quadratic forms
// are fp64, on row sums of the terms' fp64 quotients (see audit_draws_kernel); the
// edge weights and their sums are fp32.
//
// A draw's terms (r_i - r_j) w_ij are the same for every draw, so they and the
// weights are formed once per block and a draw only adds the ones of its
// completed pairs. The draws run one per lane, 32 at a time: no exchange
// between lanes, uniform (broadcast) reads of the terms and of K, and every
// lane of the fp64 pipe busy, which is what bounds the pass: about G^2 / 2 + 5 G
// fp64 operations per draw at 2 per clock and SM. Measured on one GB300, 50,000
// draws of 16 candidates with D = 4096: the call takes 104 us, its draws pass 76
// us; one block per draw, with a tree and five block reductions each, took 653 and
// 500 us. For G = 64 and 128 (3125 and 781 draws) the call takes 0.18 and 0.48
// ms, from 0.75 and 1.37 ms.
#include <math.h>

#include <type_traits>

#include "pair_coeffs_dev.cuh"

namespace pairk {
namespace {

constexpr int kAuditBlocks = 4096;  // partial-sum slots (blocks of draws), at most
constexpr int kAuditStats = 8;
constexpr int kGramThreads = 256;

// Deterministic block sum of one double per thread (all threads call).
__device__ double block_sum_double(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  for (int k = 0; k < nw; ++k) s += red[k];
  return s;
}

// K[i][j] = sum_d S[i][d] S[j][d] in fp64. Block -> a TI x TI tile of (i, j) on
// or below the diagonal; both triangles are written. One entry per block for
// G <= 32 (as many blocks as there are entries: a block's chain is D / 256
// products long, 84 -> 11 us for 16 x 4096), 4 x 4 above, where the blocks fill
// the chip anyway and a tile halves the conversions per product.
template <int TI>
__global__ void __launch_bounds__(kGramThreads)
    audit_gram_kernel(int G, int D, const float *__restrict__ S, double *K) {
  __shared__ double red[kGramThreads / 32][TI * TI];
  // Tile (ti, tj), tj <= ti, of the lower triangle in row order.
  int ti = (int)((sqrtf(8.f * blockIdx.x + 1.f) - 1.f) * 0.5f);
  while ((ti + 1) * (ti + 2) / 2 <= (int)blockIdx.x) ++ti;
  while (ti * (ti + 1) / 2 > (int)blockIdx.x) --ti;
  const int tj = (int)blockIdx.x - ti * (ti + 1) / 2;
  double acc[TI][TI];
#pragma unroll
  for (int p = 0; p < TI; ++p)
#pragma unroll
    for (int q = 0; q < TI; ++q) acc[p][q] = 0.0;
  for (int d = threadIdx.x; d < D; d += kGramThreads) {
    double x[TI], y[TI];
#pragma unroll
    for (int p = 0; p < TI; ++p) {
      const int i = min(ti * TI + p, G - 1), j = min(tj * TI + p, G - 1);
      x[p] = (double)S[(size_t)i * D + d];
      y[p] = (double)S[(size_t)j * D + d];
    }
#pragma unroll
    for (int p = 0; p < TI; ++p)
#pragma unroll
      for (int q = 0; q < TI; ++q) acc[p][q] = fma(x[p], y[q], acc[p][q]);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int p = 0; p < TI; ++p)
#pragma unroll
    for (int q = 0; q < TI; ++q) {
      double v = acc[p][q];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) red[warp][p * TI + q] = v;
    }
  __syncthreads();
  if (threadIdx.x < TI * TI) {
    double t = 0.0;
    for (int w = 0; w < kGramThreads / 32; ++w) t += red[w][threadIdx.x];
    const int i = ti * TI + threadIdx.x / TI, j = tj * TI + threadIdx.x % TI;
    if (i < G && j <= i) {
      K[(size_t)i * G + j] = t;
      K[(size_t)j * G + i] = t;
    }
  }
}

// abar, u = K abar and ||g||^2 = abar^T K abar (one block of >= G threads).
__global__ void audit_target_kernel(int G, const float *__restrict__ r, float scale,
                                    const double *__restrict__ K, double *abar, double *u,
                                    double *gg) {
  __shared__ double sa[128];
  __shared__ double red[32];
  const int i = threadIdx.x;
  const double rsum = block_sum_double(i < G ? (double)r[i] : 0.0, red);
  if (i < G) {
    sa[i] = (double)scale * 0.5 * (G * (double)r[i] - rsum);
    abar[i] = sa[i];
  }
  __syncthreads();
  double ui = 0.0;
  if (i < G) {  // K is symmetric: its columns are read, neighbours together
#pragma unroll 8
    for (int j = 0; j < G; ++j) ui += K[(size_t)j * G + i] * sa[j];
    u[i] = ui;
  }
  const double t = block_sum_double(i < G ? sa[i] * ui : 0.0, red);
  if (i == 0) *gg = t;
}

// Shared memory of the draws kernel (G x G lower triangles packed by rows,
// entry (i, j), j < i, at i (i - 1) / 2 + j; K with its diagonal).
__host__ __device__ __forceinline__ size_t audit_tri(int G) { return (size_t)G * (G - 1) / 2; }
// Warps that share 32 draws: one for G <= 32; above, a draw's fp64 operands
// (2 x 256 G bytes per 32 draws) leave room for one such batch per block only,
// and its warps divide the rows.
__host__ __device__ __forceinline__ int audit_team(int G) { return G <= 32 ? 1 : 8; }
// Warps per block: small ones of single-warp teams, so that the last round of
// blocks leaves few SMs idle (50,000 draws of 16 are 1563 batches).
__host__ __device__ __forceinline__ constexpr int audit_warps(int team) { return team == 1 ? 4 : team; }
// Whether the terms' low parts fit in shared memory too.
inline bool audit_split(int G) { return G <= 120; }
inline size_t audit_draws_smem(int G) {
  const size_t warps = audit_warps(audit_team(G)), teams = warps / audit_team(G);
  return sizeof(double) * (audit_tri(G) + G            // K
                           + 2 * (size_t)G             // abar, u
                           + teams * 2 * 32 * (size_t)G  // e, sums of a
                           + warps * 4 * 32)             // exchanges of a team
         + sizeof(float) * ((audit_split(G) ? 3 : 2) * audit_tri(G) + 2 * (size_t)G)  // terms, weights, r, pi
         + sizeof(uint32_t) * warps * 4 * 32;    // completion bits
}

template <int TW>
__device__ __forceinline__ void team_sync() {
  if constexpr (TW == 1) __syncwarp();
  else __syncthreads();
}

// Sum over the warps of a team of one value per lane (slot: 0 .. 3, its own
// exchange buffer until the team's next synchronisation with that slot).
template <int TW, typename T>
__device__ __forceinline__ T team_sum(double *xch, int slot, T v) {
  if constexpr (TW == 1) {
    return v;
  } else {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    xch[(warp * 4 + slot) * 32 + lane] = (double)v;
    __syncthreads();
    T t = (T)xch[slot * 32 + lane];
#pragma unroll
    for (int w = 1; w < TW; ++w) t += (T)xch[(w * 4 + slot) * 32 + lane];
    return t;
  }
}

__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("add.rn.f32x2 %0, %1, %2;"
      : "=l"(reinterpret_cast<unsigned long long &>(d))
      : "l"(reinterpret_cast<unsigned long long &>(a)),
        "l"(reinterpret_cast<unsigned long long &>(b)));
  return d;
}

// Draws in batches of 32, one per lane; batch q of the teams' stride. Row i of
// a batch belongs to warp i mod TW of its team. Per draw: the row sums 2 a_i =
// sum_j J_i J_j t_ij and the weight sums, then in fp64 the weighting's and flags'
// division and centring, e = a - abar, e^T K e over the lower triangle, a^T u. With a = e + abar,
// u = K abar and gg = abar^T u: a^T K a = e^T K e + 2 a^T u - gg (0 exactly where a = 0),
// formed from a itself where that leaves less than gg / 1024, as for weights or
// standardised rewards that make a small beside abar (a second pass over K, in
// batches that hold such a draw). Self-normalised coefficients are all that small,
// about 1 / C(G, 2) of abar: there a^T K a comes first and e^T K e from it, the same way.
//
// SPLIT: a term is kept as t = hi + lo, hi a multiple of q = 2^-24 times the power
// of two above G max |t|, so that fp32 sums of hi are exact in any order, and lo <=
// q / 2 the rest of the fp64 quotient: the pair is summed by one packed addition,
// and a is good to some 2^-40 of the largest term where fp32 terms and trees left
// 1e-6 of the bias, a small remainder of such sums (2.4e-6 -> 5e-8 relative, the
// rounding of scale; the draws of the size above 57 -> 73 us then). Otherwise (G > 120) fp32 terms in 16-term trees, combined
// pairwise.
template <int TW, bool SPLIT>
__global__ void __launch_bounds__(audit_warps(TW) * 32)
    audit_draws_kernel(int N, int G, const float *__restrict__ r, const float *__restrict__ rho,
                       const uint8_t *__restrict__ Jd, const double *__restrict__ wd, float scale,
                       uint32_t flags, int wmode, float w_max, const double *__restrict__ Kg,
                       const double *__restrict__ abar_g, const double *__restrict__ u_g,
                       const double *__restrict__ gg_p, double *part, int32_t *dev_err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int kWarps = audit_warps(TW), kTeams = kWarps / TW;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int team = warp / TW, tw = warp % TW;
  const int tri = (int)audit_tri(G);
  double *K = reinterpret_cast<double *>(smem_raw);
  double *abar = K + tri + G, *u = abar + G;
  double *e_all = u + G, *asum_all = e_all + kTeams * 32 * G;
  double *xch = asum_all + kTeams * 32 * G;
  using Term = std::conditional_t<SPLIT, float2, float>;
  Term *T = reinterpret_cast<Term *>(xch + kWarps * 4 * 32);
  float *Wt = reinterpret_cast<float *>(T + tri), *rs = Wt + tri, *pis = rs + G;
  uint32_t *bits_all = reinterpret_cast<uint32_t *>(pis + G);
  double *e = e_all + team * 32 * G, *asum = asum_all + team * 32 * G;
  uint32_t *bits = bits_all + team * 4 * 32;

  // ---- the group's constants (abar: what e subtracts)
  const bool small = wmode == PAIR_W_HAJEK;
  __shared__ unsigned t_max;  // bits of the largest |t|
  if (threadIdx.x == 0) t_max = 0u;
  for (int i = threadIdx.x; i < G; i += blockDim.x) {
    abar[i] = small ? 0.0 : abar_g[i];
    u[i] = u_g[i];
    rs[i] = r[i];
    pis[i] = wmode == PAIR_W_MARGINAL ? rho[(size_t)i * G + i] : 1.f;
  }
  for (int k = threadIdx.x; k < kTeams * 32 * G; k += blockDim.x) asum_all[k] = 0.0;
  __syncthreads();
  // Weight and term of pair (j, i), j < i (entry (j, i) of rho's strict upper
  // triangle). An invalid weight is NaN here and raises the error bit in the
  // draws that complete it.
  auto pair_term = [&](int j, int i, float &w) -> double {
    const double dr = (double)rs[i] - (double)rs[j];
    w = 1.f;
    if (wmode == PAIR_W_MARGINAL) {
      const bool ok = pis[i] > 0.f && pis[j] > 0.f;
      w = ok ? __frcp_rn(pis[j] * pis[i]) : __int_as_float(0x7fc00000);
      return ok ? dr / ((double)pis[j] * (double)pis[i]) : 0.0;
    }
    if (wmode == PAIR_W_UNWEIGHTED) return dr;
    const float rij = rho[(size_t)j * G + i];
    const bool ok = rij > 0.f;
    w = ok ? __frcp_rn(rij) : __int_as_float(0x7fc00000);
    if (wmode == PAIR_W_CLIPPED && w > w_max) {
      w = w_max;
      return dr * (double)w_max;
    }
    return ok ? dr / (double)rij : 0.0;
  };
  // 2^-24 of the power of two above G max |t|, and its reciprocal.
  double q = 0.0, q_inv = 0.0;
  if constexpr (SPLIT) {
    // max |t| from fp32 quotients, which round up to 3 ulp off (of the weights as
    // they are used: one rho far below 1 / w_max would else leave all terms to lo).
    float m = 0.f;
    for (int j = warp; j < G; j += kWarps)
      for (int i = j + 1 + lane; i < G; i += 32) {
        float t = fabsf(rs[i] - rs[j]);
        if (wmode == PAIR_W_MARGINAL) {
          if (pis[i] > 0.f && pis[j] > 0.f) t = __fdividef(t, pis[j] * pis[i]);
        } else if (wmode != PAIR_W_UNWEIGHTED) {
          const float rij = rho[(size_t)j * G + i];
          if (rij > 0.f) {
            const float w = __frcp_rn(rij);
            t *= wmode == PAIR_W_CLIPPED ? fminf(w, w_max) : w;
          }
        }
        m = fmaxf(m, t);
      }
    atomicMax(&t_max, __float_as_uint(m));
    __syncthreads();
    const double top = 1.000001 * (double)G * (double)__uint_as_float(t_max);
    if (top > 1e-30 && top < 1e38) {
      int e;
      frexp(top, &e);
      q = ldexp(1.0, e - 24);
      q_inv = ldexp(1.0, 24 - e);
    }
  }
  for (int j = warp; j < G; j += kWarps) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int i = j + lane + 32 * c;
      if (i >= G) continue;
      K[i * (i + 1) / 2 + j] = Kg[(size_t)j * G + i];
      if (i == j) continue;
      float w;
      const double t = pair_term(j, i, w);
      Term &o = T[i * (i - 1) / 2 + j];
      if constexpr (SPLIT) {
        // (Where no q serves, the largest term being 0, tiny or beyond fp32's range
        // over G, hi is t itself.)
        const double hi = q > 0.0 ? rint(t * q_inv) * q : (double)(float)t;
        o = make_float2((float)hi, isfinite((float)hi) ? (float)(t - hi) : 0.f);
      } else {
        o = (float)t;
      }
      Wt[i * (i - 1) / 2 + j] = w;
    }
  }
  __syncthreads();
  const double gg = *gg_p, w_all = 1.0 / (double)N;

  double acc[6] = {0, 0, 0, 0, 0, 0};  // mse, cos, vertices, edges, ess, weight (warp 0 of a team)
  const int nbatch = (int)ceil_div(N, 32);  // (N + 31 may exceed an int)
  for (int bt = blockIdx.x * kTeams + team; bt < nbatch; bt += gridDim.x * kTeams) {
    // ---- completion bits of the batch: a lane reads its own draw's flags
    // where one warp has the batch (all loads in flight; ballots, 32 candidates
    // at a time, chained 32 of them: 10 us of a batch), else by ballots.
    if constexpr (TW == 1) {
      const int b = bt * 32 + lane;
      uint32_t mw = 0u;
      if (b < N) {
        const uint8_t *row = Jd + (size_t)b * G;
#pragma unroll 16
        for (int j = 0; j < G; ++j) mw |= (row[j] != 0 ? 1u : 0u) << j;
      }
      bits[lane] = mw;
    } else {
#pragma unroll
      for (int k = 0; k < 32 / TW; ++k) {
        const int q = tw + k * TW, b = bt * 32 + q;
#pragma unroll
        for (int j0 = 0; j0 < 128; j0 += 32) {
          const bool on = b < N && j0 + lane < G && Jd[(size_t)b * G + j0 + lane] != 0;
          const uint32_t m = __ballot_sync(0xffffffffu, on);
          if (lane == 0) bits[(j0 >> 5) * 32 + q] = m;
        }
      }
    }
    team_sync<TW>();
    uint32_t m[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k * 32 < G) m[k] = bits[k * 32 + lane];
    // Whether candidate i of this lane's draw is completed.
    auto done = [&](int i) { return ((bits[(i & ~31) + lane] >> (i & 31)) & 1u) != 0u; };
    const int Kc = __popc(m[0]) + __popc(m[1]) + __popc(m[2]) + __popc(m[3]);

    // ---- row sums
    float W = 0.f, W2 = 0.f;
    double s_a = 0.0;
    for (int i = tw; i < G; i += TW) {
      const Term *row = T + i * (i - 1) / 2;
      const float *wrow = Wt + i * (i - 1) / 2;
      const bool on = done(i);
      float sw = 0.f, sw2 = 0.f;
      double a = 0.0;
      if constexpr (SPLIT) {
        float2 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = make_float2(0.f, 0.f);
#pragma unroll
        for (int blk = 0; blk < (TW == 1 ? 2 : 8); ++blk) {
          if (blk * 16 >= G) break;
          const uint32_t mb = m[blk >> 1] >> ((blk & 1) * 16);
          float wb = 0.f, wb2 = 0.f;
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const int j = blk * 16 + q;
            const bool jon = (mb >> q) & 1u;
            // Uniform over the warp: which triangle, and past the group.
            float2 t = make_float2(0.f, 0.f);
            if (j < i) {
              t = row[j];
              const float w = jon ? wrow[j] : 0.f;
              wb += w;
              wb2 = fmaf(w, w, wb2);
            } else if (j > i && j < G) {
              t = T[j * (j - 1) / 2 + i];
              t = make_float2(-t.x, -t.y);
            }
            x[q & 3] = add2(x[q & 3], make_float2(jon ? t.x : 0.f, jon ? t.y : 0.f));
          }
          sw += wb;
          sw2 += wb2;
        }
        const float2 y = add2(add2(x[0], x[1]), add2(x[2], x[3]));
        if (on) a = (double)y.x + (double)y.y;
      } else {
        float p[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int blk = 0; blk < 8; ++blk) {
          float c = 0.f;
          if (blk * 16 < G) {
            const uint32_t mb = m[blk >> 1] >> ((blk & 1) * 16);
            float x[16], wb = 0.f, wb2 = 0.f;
#pragma unroll
            for (int q = 0; q < 16; ++q) {
              const int j = blk * 16 + q;
              const bool jon = (mb >> q) & 1u;
              float t = 0.f;
              if (j < i) {
                t = row[j];
                const float w = jon ? wrow[j] : 0.f;
                wb += w;
                wb2 = fmaf(w, w, wb2);
              } else if (j > i && j < G) {
                t = -T[j * (j - 1) / 2 + i];
              }
              x[q] = jon ? t : 0.f;
            }
            sw += wb;
            sw2 += wb2;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1)
#pragma unroll
              for (int q = 0; q < o; ++q) x[q] += x[q + o];
            c = x[0];
          }
          int mm = blk;
#pragma unroll
          for (int l = 0; l < 4; ++l) {
            if (mm & 1) { c = p[l] + c; mm >>= 1; }
            else { p[l] = c; break; }
          }
        }
        if (on) a = (double)p[3];
      }
      if (on) {
        W += sw;
        W2 += sw2;
      }
      s_a += a;
      e[i * 32 + lane] = a;
    }
    W = team_sum<TW>(xch, 0, W);
    W2 = team_sum<TW>(xch, 1, W2);
    if (W != W) flag_error(dev_err, PAIR_DEV_ERR_NONPOSITIVE_INCLUSION);

    // ---- the divisions, the centring and the scale of the coefficients:
    // a_i -> f (a_i - mean), a half of f being the row sums'
    double f = 0.5 * (double)scale;
    if (wmode == PAIR_W_HAJEK) f = W > 0.f ? f / (double)W : 0.0;
    if ((flags & PAIR_STANDARDIZE) && Kc >= 2) {
      double sr = 0.0, ss = 0.0;
      for (int i = 0; i < G; ++i) sr += done(i) ? (double)rs[i] : 0.0;
      const double mean = sr / (double)Kc;
      for (int i = 0; i < G; ++i) {
        const double dv = done(i) ? (double)rs[i] - mean : 0.0;
        ss = fma(dv, dv, ss);
      }
      const double sd = sqrt(ss / (double)(Kc - 1));
      f = sd > 0.0 ? f / sd : 0.0;
    }
    double mean_a = 0.0;
    if (flags & PAIR_CENTER) {
      s_a = team_sum<TW>(xch, 2, s_a);
      mean_a = Kc > 0 ? s_a / (double)Kc : 0.0;
    }

    // ---- fp64: e = a - abar (small: a itself), the sums of a, a^T u (before its factor)
    const int b = bt * 32 + lane;
    const double w = b < N ? (wd ? wd[b] : w_all) : 0.0, wf = w * f;
    double au = 0.0;
    bool any = false;  // (of a before its factor; f = 0 is checked below)
    for (int i = tw; i < G; i += TW) {
      double a = e[i * 32 + lane];
      if ((flags & PAIR_CENTER) && done(i)) a -= mean_a;
      any |= a != 0.0;
      e[i * 32 + lane] = fma(a, f, -abar[i]);
      asum[i * 32 + lane] = fma(wf, a, asum[i * 32 + lane]);
      au = fma(a, u[i], au);
    }
    team_sync<TW>();

    // ---- x^T K x over the lower triangle
    auto form = [&](auto x) {
      double q = 0.0;
      for (int i = tw; i < G; i += TW) {
        const double *row = K + i * (i + 1) / 2;
        double s0 = 0.0, s1 = 0.0;
        int j = 0;
        for (; j + 4 <= i; j += 4) {
          s0 = fma(row[j], x(j), s0);
          s1 = fma(row[j + 1], x(j + 1), s1);
          s0 = fma(row[j + 2], x(j + 2), s0);
          s1 = fma(row[j + 3], x(j + 3), s1);
        }
        for (; j < i; ++j) s0 = fma(row[j], x(j), s0);
        const double xi = x(i);
        q = fma(xi, fma(2.0, s0 + s1, row[i] * xi), q);
      }
      return team_sum<TW>(xch, 2, q);
    };
    const double p = form([&](int j) { return e[j * 32 + lane]; });
    au = team_sum<TW>(xch, 3, au) * f;
    if constexpr (TW > 1) any = team_sum<TW>(xch, 0, any ? 1.f : 0.f) > 0.f;
    any = any && f != 0.0;
    // The other of the two forms (the conditions are the same in every warp of the team).
    const double sign = small ? -1.0 : 1.0;
    double other = fma(sign, fma(2.0, au, -gg), p);
    const bool redo = (any || small) && other < gg * 0x1p-10;
    if (__any_sync(0xffffffffu, redo)) {
      const double x = form([&](int j) { return fma(sign, abar_g[j], e[j * 32 + lane]); });
      if (redo) other = x;
    }
    const double q = small ? other : p, q_aa = !any ? 0.0 : small ? p : other;
    if (tw == 0) {
      const double q_au = any ? au : 0.0;
      const double cosb = (q_aa > 0.0 && gg > 0.0) ? q_au * rsqrt(q_aa * gg) : 0.0;
      const double ess = W2 > 0.f ? (double)W * (double)W / (double)W2 : 0.0;
      acc[0] = fma(w, q, acc[0]);
      acc[1] = fma(w, cosb, acc[1]);
      acc[2] = fma(w, (double)Kc, acc[2]);
      acc[3] = fma(w, (double)(Kc * (Kc - 1) / 2), acc[3]);
      acc[4] = fma(w, ess, acc[4]);
      acc[5] += w;
    }
    team_sync<TW>();  // bits, e and the exchanges are rewritten by the next batch
  }

  // ---- the block's partial sums, lanes then teams in order
  double *pq = part + (size_t)blockIdx.x * (kAuditStats + G);
#pragma unroll
  for (int k = 0; k < 6; ++k)
    for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
  __syncthreads();
  if (tw == 0 && lane == 0)
#pragma unroll
    for (int k = 0; k < 6; ++k) xch[team * 6 + k] = acc[k];
  __syncthreads();
  if (threadIdx.x < 6) {
    double t = 0.0;
    for (int q = 0; q < kTeams; ++q) t += xch[q * 6 + threadIdx.x];
    pq[threadIdx.x] = t;
  }
  for (int i = warp; i < G; i += kWarps) {
    double t = 0.0;
    for (int q = 0; q < kTeams; ++q) t += asum_all[((size_t)q * G + i) * 32 + lane];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) pq[kAuditStats + i] = t;
  }
}

// Sums the partials (each column by one warp, lanes over the blocks, then a
// butterfly: a fixed order), normalises by the total weight, and forms the
// bias E[a] - abar, its norm through K and (optionally) the vector (E[a] -
// abar) S. Every block forms the means; block 0 writes the statistics, and
// the blocks share the D components of the bias (one block for all of it
// took 95 us at 16 x 4096).
__global__ void __launch_bounds__(256)
    audit_finish_kernel(int nblk, int G, int D, const float *__restrict__ S,
                        const double *__restrict__ K, const double *__restrict__ abar,
                        const double *__restrict__ gg_p, const double *__restrict__ part,
                        double *stats, double *bias) {
  __shared__ double em[128];
  __shared__ double red[32];
  __shared__ double tot[6];
  const int tid = threadIdx.x, lane = tid & 31;
  const int stride = kAuditStats + G;
  for (int k = tid >> 5; k < 6 + G; k += 8) {
    const int col = k < 6 ? k : kAuditStats + (k - 6);
    double s = 0.0;
    for (int q = lane; q < nblk; q += 32) s += part[(size_t)q * stride + col];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      if (k < 6) tot[k] = s;
      else em[k - 6] = s;
    }
  }
  __syncthreads();
  const double W = tot[5];
  if (tid < G) em[tid] = (W > 0.0 ? em[tid] / W : 0.0) - abar[tid];
  __syncthreads();
  if (blockIdx.x == 0) {
    double Ke = 0.0;
    if (tid < G)
#pragma unroll 8
      for (int j = 0; j < G; ++j) Ke += K[(size_t)j * G + tid] * em[j];
    const double bb = block_sum_double(tid < G ? em[tid] * Ke : 0.0, red);
    if (tid == 0) {
      stats[0] = sqrt(bb > 0.0 ? bb : 0.0);
      for (int k = 0; k < 5; ++k) stats[1 + k] = W > 0.0 ? tot[k] / W : 0.0;
      stats[6] = *gg_p;
      stats[7] = W;
    }
  }
  if (bias)
    for (int d = blockIdx.x * 256 + tid; d < D; d += gridDim.x * 256) {
      double s = 0.0;
#pragma unroll 8
      for (int i = 0; i < G; ++i) s += em[i] * (double)S[(size_t)i * D + d];
      bias[d] = s;
    }
}

template <int TW, bool SPLIT>
pair_status launch_draws(int &nblk, int nsm, size_t smem, int N, int G, const float *r, const float *rho,
                         const uint8_t *Jd, const double *wd, float scale, uint32_t flags,
                         int wmode, float w_max, const double *K, const double *abar,
                         const double *u, const double *gg, double *part, int32_t *dev_err,
                         cudaStream_t s) {
  PAIR_CUDA_TRY(cudaFuncSetAttribute(audit_draws_kernel<TW, SPLIT>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  // One batch of 32 draws per team as far as the chip holds the blocks at once (and
  // the partial slots); a stride over the batches beyond that.
  int per_sm = 0;
  PAIR_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &per_sm, audit_draws_kernel<TW, SPLIT>, audit_warps(TW) * 32, smem));
  const int64_t want = ceil_div(ceil_div(N, 32), audit_warps(TW) / TW);
  const int64_t most = (int64_t)nsm * (per_sm > 0 ? per_sm : 1);
  nblk = (int)(want < most ? want : most);
  if (nblk > kAuditBlocks) nblk = kAuditBlocks;
  PAIR_BEGIN("audit_draws", s);
  audit_draws_kernel<TW, SPLIT><<<nblk, audit_warps(TW) * 32, smem, s>>>(
      N, G, r, rho, Jd, wd, scale, flags, wmode, w_max, K, abar, u, gg, part, dev_err);
  PAIR_LAUNCH_CHECK(s);
  return PAIR_OK;
}

pair_status launch_audit(int N, int G, int D, const float *r, const float *rho, const float *S,
                         const uint8_t *Jd, const double *wd, float scale, uint32_t flags,
                         int wmode, float w_max, double *stats, double *bias, double *ws,
                         int32_t *dev_err, cudaStream_t s) {
  double *K = ws, *abar = K + (size_t)G * G, *u = abar + G, *gg = u + G;
  double *part = gg + 2;
  const int gt = G <= 32 ? G : (G + 3) / 4;  // rows of gram tiles
  PAIR_BEGIN("audit_gram", s);
  if (G <= 32)
    audit_gram_kernel<1><<<gt * (gt + 1) / 2, kGramThreads, 0, s>>>(G, D, S, K);
  else
    audit_gram_kernel<4><<<gt * (gt + 1) / 2, kGramThreads, 0, s>>>(G, D, S, K);
  PAIR_LAUNCH_CHECK(s);
  PAIR_BEGIN("audit_target", s);
  audit_target_kernel<<<1, 128, 0, s>>>(G, r, scale, K, abar, u, gg);
  PAIR_LAUNCH_CHECK(s);
  int dev = 0, nsm = 0, nblk = 0;
  PAIR_CUDA_TRY(cudaGetDevice(&dev));
  PAIR_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const size_t smem = audit_draws_smem(G);
  pair_status st;
  if (audit_team(G) == 1)
    st = launch_draws<1, true>(nblk, nsm, smem, N, G, r, rho, Jd, wd, scale, flags, wmode, w_max, K, abar,
                               u, gg, part, dev_err, s);
  else if (audit_split(G))
    st = launch_draws<8, true>(nblk, nsm, smem, N, G, r, rho, Jd, wd, scale, flags, wmode, w_max, K, abar,
                               u, gg, part, dev_err, s);
  else
    st = launch_draws<8, false>(nblk, nsm, smem, N, G, r, rho, Jd, wd, scale, flags, wmode, w_max, K,
                                abar, u, gg, part, dev_err, s);
  if (st != PAIR_OK) return st;
  PAIR_BEGIN("audit_finish", s);
  const int fin = bias ? (int)ceil_div(D, 256) : 1;
  audit_finish_kernel<<<fin < nsm ? fin : nsm, 256, 0, s>>>(nblk, G, D, S, K, abar, gg, part,
                                                            stats, bias);
  PAIR_LAUNCH_CHECK(s);
  return PAIR_OK;
}

}  // namespace
}  // namespace pairk

using namespace pairk;

extern "C" size_t pair_audit_workspace_size(int32_t N, int32_t G, int32_t D) {
  if (N < 1 || G < 2 || G > PAIR_MAX_G || D < 1) return 0;
  const int GP = G <= 32 ? 32 : G <= 64 ? 64 : 128;
  const size_t nblk = N < kAuditBlocks ? (size_t)N : (size_t)kAuditBlocks;
  return sizeof(double) * ((size_t)G * G + 2 * (size_t)G + 2 + nblk * (kAuditStats + GP));
}

extern "C" pair_status pair_audit(int32_t N, int32_t G, int32_t D, const float *r,
                                  const float *rho, const float *S, const uint8_t *Jdraws,
                                  const double *draw_weight, float scale, uint32_t flags,
                                  pair_weighting wmode, float w_max, double *stats, double *bias,
                                  void *ws, size_t ws_bytes, int32_t *dev_err,
                                  pair_stream_t stream) {
  reset_launches();
  const size_t need = pair_audit_workspace_size(N, G, D);
  if (need == 0 || !r || !S || !Jdraws || !stats ||
      (flags & ~(PAIR_CENTER | PAIR_STANDARDIZE)) != 0)
    return PAIR_ERR_INVALID_ARG;
  const int wm = (int)wmode;
  if (wm < PAIR_W_HT || wm > PAIR_W_HAJEK) return PAIR_ERR_INVALID_ARG;
  if (wm != PAIR_W_UNWEIGHTED && !rho) return PAIR_ERR_INVALID_ARG;
  if (wm == PAIR_W_CLIPPED && !(w_max > 0.f && w_max <= 3.0e38f)) return PAIR_ERR_INVALID_ARG;
  if (!ws || ws_bytes < need || (reinterpret_cast<uintptr_t>(ws) & 15u)) return PAIR_ERR_WORKSPACE;
  const pair_status dv = check_device();
  if (dv != PAIR_OK) return dv;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  return launch_audit(N, G, D, r, rho, S, Jdraws, draw_weight, scale, flags, wm, w_max, stats,
                      bias, static_cast<double *>(ws), dev_err, s);
}
