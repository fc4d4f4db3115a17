// pair_allocate: the allocation step before the path (Sec. 4.3-4.4). For
// every group, the contrast graph (Eq. disagreement / Eq. edge-proxy), the
// shared-vertex surrogate b_i (Sec. 4.4) and the continuation probabilities
// of the convex program of Eqs. (convex-objective)-(budget):
//     min_x  Phi(x) = sum_{i<j} a_ij e^(x_i + x_j) + sum_i b_i e^(x_i)
//     s.t.   sum_i c_i e^(-x_i) <= budget,   0 <= x_i <= -log pi_min,
// with pi_i = e^(-x_i).
//
// Solver (one CTA per group, fp64), in the variables pi: with v_i = 1 / pi_i
// the program is
//     min  Phi = sum_{i<j} a_ij v_i v_j + sum_i b_i v_i
//     s.t. sum_i c_i pi_i = budget,   pi_min <= pi_i <= 1,
// still convex, and with linear constraints only (Phi falls in every pi_i, so
// the budget is spent; kBudgetMargin keeps the rounded sum below it). It is
// solved by a primal-dual interior-point method with Mehrotra's predictor and
// corrector: about 8 to 11 steps to a duality gap of 1e-12 Phi, where a
// log-barrier Newton iteration in x took 47 (groups of 16) and 80 (64).
//
// The Newton system in the relative steps d_i = dpi_i / pi_i is
//     M_ij = a_ij v_i v_j (i != j),
//     M_ii = 2 v_i (w_i + b_i) + pi_i^2 (zl_i / sl_i + zh_i / sh_i),
// w = A v. Its off-diagonal row sum is v_i w_i, at most half its diagonal (and
// about 1 / 2G of it for a dense graph, where b_i is about G sum_j a_ij), so
// no factorisation is needed: Chebyshev's iteration on the system scaled by
// its diagonal, whose spectrum lies within rho = max_i v_i w_i / M_ii <= 1/2 of
// 1, gains a factor of at least 3.7 per product with A. A reduction to a tenth is
// enough as long as whole steps pass the test of the residuals: what the solve
// leaves is in the next step's residual, and the steps are as many as with 1e-12
// (10.3 against 9.8 on groups of 64). So rho <= 1/10, every dense group of 16 or
// more, needs no product at all: the step solves the diagonal. Where rho is near
// 1/2 (groups of 2, sparse graphs) a direction a tenth off can fail that test again
// and again; its halved steps then stand still (45 of 100,000 groups of 2 and a few
// of 100,000 sparse ones of 3 to 8 reached the cap of steps). So from a group's
// second halving on its systems are solved to 1e-6: none of a million groups each
// of 2, 3, 4, 5 and 8, dense and sparse, took more than 20 steps then. (A first
// halving alone says little: switching there cost 4096 groups of 64, a tenth of
// which have one, 2.93 instead of 2.45 ms.)
// Odd degrees only: their residual polynomial vanishes at 1, where the
// coordinates at a bound lie, so those are exact (even degrees stall there). The
// stopping test is on the fp64 residuals themselves.
//
// A vertex without an edge has no curvature but its complementarity's, z / s: once
// that has shrunk below its dual residual its step points far outside the box and
// the rest stands still. So after two halvings the corrector's second-order term,
// which such a step makes as large as the step, is scaled by the predictor's step
// lengths, and the centring keeps the gap from falling behind the residual
// (kGapBehind). Without the two up to 2039 of 40,000 groups of 6 with such vertices
// and costs over decades stopped at the cap. With them all of 9.2 million groups of 2
// to 64 were solved (dense, sparse, uneven, with such vertices; costs up to exp(6 N);
// half of them within 1e-6 to 1/2 of the budget's limits), two of them in more than 80
// steps; the log-barrier form left 12 at its cap.
//
// What bounds it: the fp64 pipe (2 multiply-adds per clock and SM) for many
// groups, the chain of a step's exchanges for few. Measured on one GB300,
// against the factorising log-barrier form: 64 groups of 16 in 0.078 ms (2.43
// ms), 4096 groups of 64 in 2.45 ms (178 ms); with a root per
// entry of A 2.70 ms, with kLinRel = 1e-3 too 0.107 and 4.79 ms, with IEEE divisions in place of rcp_approx / rcp_newton and full
// butterflies besides 0.188 and 6.84 ms.
//
// The paper solves the same program with SLSQP on the CPU (App. C); any
// method reaching its optimum is equivalent. Cases the program leaves without
// an interior (budget >= sum c: pi = 1; budget = pi_min sum c: pi = pi_min;
// budget below that: infeasible) and the flat objective (all a_ij = b_i = 0)
// are classified first, from the fp64 sum of c in index order. If the
// iteration does not converge within its cap, the group falls back to the
// uniform pi = budget / sum c of the same expected cost (the paper's
// fallback).
#include <math.h>
#include <stdint.h>

#include "pair_common.cuh"

namespace pairk {
namespace {

constexpr int kAllocMaxSteps = 200;     // interior-point steps per group (most take 6 to 17)
constexpr int kAllocMaxBacktrack = 20;  // halvings of one step
constexpr double kGapRel = 1e-12;       // stop at gap <= kGapRel * Phi (and the dual residual)
// The budget the equality constraint aims at is this much (relative) below
// the caller's: the rounding of the fp64 sum of c pi (at most 128 2^-53) and
// the primal residual allowed at the end (kPrimalRel) then never spend more.
constexpr double kBudgetMargin = 4e-14;
constexpr double kPrimalRel = 2e-14;
constexpr float kLinRel = 0.1f;     // reduction of the Newton system's residual,
constexpr float kLinTight = 1e-6f;  // and from a group's second halving on
// Rounding of the dual residual: its terms y c pi sum to y budget, which exceeds
// Phi by many powers of ten where costs do and the budget is near pi_min sum c.
// The residual then stops there, above kGapRel Phi (5 to 17 of 20,000 such groups
// reached the cap of steps; the log-barrier form, which has no such test, at most 3).
constexpr double kDualRound = 8e-16;
constexpr int kLinMaxDegree = 61;   // reached only if rounding puts rho far above 1/2
constexpr double kGapBehind = 10.0; // times the gap: a dual residual above it is
constexpr double kGapHold = 3e-3;   // answered by a complementarity of this part of it
constexpr float kStepFrac = 0.995f; // of the largest step that keeps the interior
constexpr double kStartMu = 0.1;    // the start's complementarity: kStartMu Phi in all

// Where a value only steers (step lengths, the centring parameter) or enters
// both sides of an identity (the slacks' reciprocals), rcp_approx stands in for
// a division; v and the diagonal's inverse take rcp_newton.

// Shape of a group's CTA: GP >= G is the padded group size, TPR adjacent
// threads share a row of A and each holds its coordinate's state.
template <int GP>
struct AllocShape {
  static constexpr int kThreads = GP <= 16 ? 32 : 2 * GP;
  static constexpr int kTpr = kThreads / GP;
  static constexpr int kWarps = kThreads / 32;
  // Blocks per SM that the register allocation leaves room for: what shared
  // memory holds of groups of 64; elsewhere the compiler's choice (0; asking for
  // 16 warps of the small groups cost 81 us instead of 78 on 64 x 16).
  static constexpr int kBlocks = GP == 64 ? 5 : 0;
};

// Row pitch of A (odd: rows start in different shared-memory banks).
__host__ __device__ __forceinline__ int alloc_pitch(int G) { return G | 1; }

template <int GP>
struct AllocSmem {
  double x[2][2][GP];  // operands of a product: [buffer][right-hand side]
  double red[2][4][AllocShape<GP>::kWarps];
  float redm[2][2][AllocShape<GP>::kWarps];
  double c[GP];
  float p[GP], m[GP];
  double sum_c;
  int any;
};

template <int GP>
__device__ __forceinline__ void alloc_sync() {
  if constexpr (AllocShape<GP>::kWarps == 1) __syncwarp();
  else __syncthreads();
}

// One group's CTA: its thread's coordinate (i, replicated over the TPR
// threads of the row), and the exchanges.
template <int GP>
struct AllocGroup {
  static constexpr int kTpr = AllocShape<GP>::kTpr;
  static constexpr int kWarps = AllocShape<GP>::kWarps;
  AllocSmem<GP> &sm;
  double *A;  // [G][pitch], zero diagonal
  int G, pitch, i, sub;
  bool act;
  int xb, rb;  // buffers of the next product and the next reduction
  float lin;   // reduction of a system's residual

  // NS sums (fp64) and NM maxima (fp32: they only steer) over the group's
  // coordinates, to every thread. The replicas of a coordinate hold the same
  // value, so the butterfly starts at the row distance. Its first stages
  // halve the number of sums a lane carries (4 sums over 16 lanes take 5
  // additions instead of 16), and shuffles hand the totals back. Two buffers:
  // a reduction is one barrier.
  template <int NS, int NM>
  __device__ void reduce(double (&v)[NS], float (&mx)[NM]) {
    const int lane = threadIdx.x & 31;
    constexpr int H1 = NS >= 3 ? 2 : 1;  // sums a lane keeps after the first stage
    double t[NS >= 3 ? 2 : 1];
    int o = kTpr;
    if constexpr (NS >= 2) {
      const bool up = lane & o;
#pragma unroll
      for (int k = 0; k < H1; ++k) {
        const double hi = k + H1 < NS ? v[k + H1] : 0.0;
        const double keep = up ? hi : v[k], send = up ? v[k] : hi;
        t[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
      o <<= 1;
    } else {
      t[0] = v[0];
    }
    if constexpr (NS >= 3) {
      const bool up = lane & o;
      const double keep = up ? t[1] : t[0], send = up ? t[0] : t[1];
      t[0] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      o <<= 1;
    }
    for (; o < 32; o <<= 1) t[0] += __shfl_xor_sync(0xffffffffu, t[0], o);
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      // Sum k ended in the lanes whose halving bits spell it.
      const int src = NS >= 3 ? (k / 2) * kTpr + (k % 2) * 2 * kTpr : k * kTpr;
      v[k] = __shfl_sync(0xffffffffu, t[0], src);
    }
#pragma unroll
    for (int q = kTpr; q < 32; q <<= 1)
#pragma unroll
      for (int k = 0; k < NM; ++k) mx[k] = fmaxf(mx[k], __shfl_xor_sync(0xffffffffu, mx[k], q));
    if constexpr (kWarps > 1) {
      if (lane == 0) {
#pragma unroll
        for (int k = 0; k < NS; ++k) sm.red[rb][k][threadIdx.x >> 5] = v[k];
#pragma unroll
        for (int k = 0; k < NM; ++k) sm.redm[rb][k][threadIdx.x >> 5] = mx[k];
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        v[k] = sm.red[rb][k][0];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) v[k] += sm.red[rb][k][w];
      }
#pragma unroll
      for (int k = 0; k < NM; ++k) {
        mx[k] = sm.redm[rb][k][0];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) mx[k] = fmaxf(mx[k], sm.redm[rb][k][w]);
      }
      rb ^= 1;
    }
  }
  template <int NS>
  __device__ void sum(double (&v)[NS]) {
    float none[1] = {0.f};
    reduce<NS, 1>(v, none);
  }

  // y_r = (A x_r)_i for NR right-hand sides, x given per coordinate.
  template <int NR>
  __device__ void product(const double (&x)[NR], double (&y)[NR]) {
    if (sub == 0)
#pragma unroll
      for (int r = 0; r < NR; ++r) sm.x[xb][r][i] = act ? x[r] : 0.0;
    alloc_sync<GP>();
    double acc[NR][2];
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r][0] = acc[r][1] = 0.0;
    if (act) {
      const double *row = A + (size_t)i * pitch;
      int j = sub;
      for (; j + 3 * kTpr < G; j += 4 * kTpr) {
        double a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = row[j + u * kTpr];
#pragma unroll
        for (int r = 0; r < NR; ++r)
#pragma unroll
          for (int u = 0; u < 4; ++u)
            acc[r][u & 1] = fma(a[u], sm.x[xb][r][j + u * kTpr], acc[r][u & 1]);
      }
      for (; j < G; j += kTpr) {
        const double a = row[j];
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[r][0] = fma(a, sm.x[xb][r][j], acc[r][0]);
      }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      double t = acc[r][0] + acc[r][1];
#pragma unroll
      for (int o = 1; o < kTpr; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      y[r] = t;
    }
    xb ^= 1;
  }

  // Approximate solutions of M x_r = rhs_r (see the head of this file):
  // Chebyshev's iteration on M scaled by its diagonal (inverse rd), odd
  // degree, until the residual is reduced by lin.
  template <int NR>
  __device__ void solve(double v, double rd, float rho, const double (&rhs)[NR],
                        double (&x)[NR]) {
    double r[NR], d[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      r[k] = d[k] = x[k] = rhs[k] * rd;
    }
    if (!(rho > 0.f)) return;
    // err = 1 / T_n(1 / rho) by its recurrence r1 = 1 / (2 / rho - r0). The
    // two coefficients of an update are r1 r0 and 2 r1 / rho = 1 + r1 r0; in
    // the second form an odd degree vanishes at 1 whatever r1's rounding.
    const float s = 1.f / rho;
    float r0 = rho, err = rho;
    const double vrd = v * rd;
    for (int n = 1; !(err <= lin && (n & 1)) && n < kLinMaxDegree; ++n) {
      double t[NR], y[NR];
#pragma unroll
      for (int k = 0; k < NR; ++k) t[k] = v * d[k];
      product<NR>(t, y);
      const float r1 = 1.f / (2.f * s - r0);
      const double al = (double)(r1 * r0);
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        r[k] -= fma(vrd, y[k], d[k]);
        d[k] = fma(al, d[k] + r[k], r[k]);
        x[k] += d[k];
      }
      r0 = r1;
      err *= r0;
    }
  }
};

// Edge proxy a_ij: the explicit array, else Eq. (disagreement) from p_hat,
// times ((m_i + m_j) / 2)^2 with score-norm predictions (Eq. edge-proxy).
__device__ __forceinline__ double edge_proxy(float pi_, float pj_, bool norms, float mi,
                                             float mj) {
  const double pi = pi_, pj = pj_;
  double d = pi * (1.0 - pj) + (1.0 - pi) * pj;
  if (norms) {
    const double h = 0.5 * ((double)mi + (double)mj);
    d *= h * h;
  }
  return d;
}

template <int GP>
__global__ void __launch_bounds__(AllocShape<GP>::kThreads, AllocShape<GP>::kBlocks)
    alloc_kernel(int G, const float *__restrict__ p_hat, const float *__restrict__ m_hat,
                 const float *__restrict__ a, const float *__restrict__ c_hat,
                 const float *__restrict__ budget_in, float pi_min, float *__restrict__ pi_out,
                 double *__restrict__ stats, int32_t *dev_err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int kTpr = AllocShape<GP>::kTpr;
  AllocSmem<GP> &sm = *reinterpret_cast<AllocSmem<GP> *>(smem_raw);
  const int i = threadIdx.x / kTpr, sub = threadIdx.x % kTpr, g = blockIdx.x;
  const bool act = i < G;
  AllocGroup<GP> grp{sm, reinterpret_cast<double *>(smem_raw + sizeof(AllocSmem<GP>)),
                     G,  alloc_pitch(G), i, sub, act, 0, 0, kLinRel};

  // ---- inputs and their validity
  bool bad = false;
  double ci = 1.0;
  if (act) {
    ci = (double)c_hat[(size_t)g * G + i];
    bad |= !(ci > 0.0 && ci <= 3.0e38);
    if (!a) {
      const float pf = p_hat[(size_t)g * G + i];
      bad |= !(pf >= 0.f && pf <= 1.f);
      sm.p[i] = pf;
      if (m_hat) {
        const float mf = m_hat[(size_t)g * G + i];
        bad |= !(mf >= 0.f && mf <= 3.0e38f);
        sm.m[i] = mf;
      }
    } else {
      for (int j = sub; j < G; j += kTpr) {
        const float v = a[((size_t)g * G + i) * G + j];
        bad |= (j != i) && !(v >= 0.f && v <= 3.0e38f);
      }
    }
    sm.c[i] = ci;
  }
  const double budget = (double)budget_in[g];
  bad |= !(budget > 0.0 && budget <= 3.0e38);
  if (threadIdx.x == 0) sm.any = 0;
  alloc_sync<GP>();
  if (bad) atomicOr(&sm.any, 1);
  // The sum of c in index order (the classification is bit-identical to a
  // sequential fp64 sum on the host).
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < G; ++k) s += sm.c[k];
    sm.sum_c = s;
  }
  alloc_sync<GP>();
  const bool invalid = sm.any != 0;
  const double sc = sm.sum_c, pmin = (double)pi_min;

  // ---- A and b_i = (sum_{j != i} sqrt a_ij)^2 - sum_{j != i} a_ij. The
  // proxies from predictions are symmetric: row i forms the pairs (i, i + s mod
  // G) for s up to G / 2, a_ij at [j][i] and its square root at [i][j] until the
  // rows are summed (a square root is some twenty fp64 instructions: 2.70 -> 2.45
  // ms on 4096 groups of 64). Groups of up to 32, where the extra passes cost as
  // much, and an explicit array take every entry by itself.
  double bi = 0.0, asum = 0.0, sq = 0.0;
  if (GP <= 32 || a) {
    if (act && !invalid) {
      const float pi_ = a ? 0.f : sm.p[i], mi = m_hat && !a ? sm.m[i] : 0.f;
      for (int j = sub; j < G; j += kTpr) {
        double v = 0.0;
        if (j != i)
          v = a ? (double)a[((size_t)g * G + i) * G + j]
                : edge_proxy(pi_, sm.p[j], m_hat != nullptr, mi, m_hat ? sm.m[j] : 0.f);
        grp.A[(size_t)i * grp.pitch + j] = v;
        sq += sqrt(v);
        asum += v;
      }
    }
  } else {
    const float pi_ = act ? sm.p[i] : 0.f, mi = act && m_hat ? sm.m[i] : 0.f;
    // Row i's pairs: s = 1 .. half (the pairs half the group apart belong to
    // the first half of the rows).
    const int half = G % 2 == 0 && i >= G / 2 ? G / 2 - 1 : G / 2;
    if (act && !invalid) {
      if (sub == 0) grp.A[(size_t)i * grp.pitch + i] = 0.0;
      for (int s = 1 + sub; s <= half; s += kTpr) {
        const int j = i + s < G ? i + s : i + s - G;
        const double v =
            edge_proxy(pi_, sm.p[j], m_hat != nullptr, mi, m_hat ? sm.m[j] : 0.f);
        grp.A[(size_t)j * grp.pitch + i] = v;
        grp.A[(size_t)i * grp.pitch + j] = sqrt(v);
      }
    }
    alloc_sync<GP>();
    if (act && !invalid)
      for (int s = 1 + sub; s < G; s += kTpr) {
        const int j = i + s < G ? i + s : i + s - G;
        const double x = grp.A[(size_t)i * grp.pitch + j], y = grp.A[(size_t)j * grp.pitch + i];
        const bool root = s <= half;  // [i][j] holds the root, [j][i] the proxy
        sq += root ? x : y;
        asum += root ? y : x;
      }
    alloc_sync<GP>();
    if (act && !invalid)
      for (int s = 1 + sub; s <= half; s += kTpr) {
        const int j = i + s < G ? i + s : i + s - G;
        grp.A[(size_t)i * grp.pitch + j] = grp.A[(size_t)j * grp.pitch + i];
      }
  }
#pragma unroll
  for (int o = 1; o < kTpr; o <<= 1) {
    sq += __shfl_xor_sync(0xffffffffu, sq, o);
    asum += __shfl_xor_sync(0xffffffffu, asum, o);
  }
  bi = sq * sq - asum;
  bool flat;
  {
    double v[1] = {act ? asum + bi : 0.0};
    grp.template sum<1>(v);
    flat = v[0] == 0.0;
  }

  int status;
  if (invalid) status = PAIR_ALLOC_INVALID;
  else if (budget >= sc) status = PAIR_ALLOC_SLACK;
  else if (budget == pmin * sc) status = PAIR_ALLOC_FLOOR;
  else if (budget < pmin * sc) status = PAIR_ALLOC_INFEASIBLE;
  else if (flat) status = PAIR_ALLOC_FLAT;
  else status = PAIR_ALLOC_OK;

  double pi = 1.0, gap = 0.0, phi = 0.0, spent = 0.0;
  int steps = 0, halvings = 0;
  bool solved = false;
  if (status == PAIR_ALLOC_OK) {
    const double target = budget - fmin(kBudgetMargin * budget, 0.5 * (budget - pmin * sc));
    pi = target / sc;  // uniform start
    double sl = pi - pmin, sh = 1.0 - pi;
    if (!(sl > 0.0 && sh > 0.0)) sl = sh = 0.0;  // no interior in fp64: fall back
    const double half_inv = 0.5 / G;
    double v = rcp_newton(pi), w, zl, zh, y, dres;
    float rho;
    {
      double x[1] = {v}, r[1];
      grp.template product<1>(x, r);
      w = r[0];
      const double wb = w + bi;
      double s[3] = {act ? v * (0.5 * w + bi) : 0.0, act ? v * wb : 0.0, act ? ci * pi : 0.0};
      grp.template sum<3>(s);
      phi = s[0];
      y = s[1] / s[2];
      zl = kStartMu * phi * half_inv / sl;
      zh = kStartMu * phi * half_inv / sh;
    }
    // At a point: the sums Phi, duality gap, dual residual and cost, the
    // inverse diagonal rd of M, and rho.
    double rsl, rsh, rd;
    auto measure = [&](double pi, double v, double w, double sl, double sh, double zl, double zh,
                       double y, double (&s)[4], float &rho) {
      const double vw = v * w, vwb = fma(v, bi, vw), cp = ci * pi;
      rsl = rcp_approx(sl);
      rsh = rcp_approx(sh);
      rd = rcp_newton(fma(pi * pi, zl * rsl + zh * rsh, 2.0 * vwb));
      s[0] = act ? vwb - 0.5 * vw : 0.0;
      s[1] = act ? zl * sl + zh * sh : 0.0;
      s[2] = act ? fabs(fma(y, cp, -vwb) - (zl - zh) * pi) : 0.0;
      s[3] = act ? cp : 0.0;
      float m[1] = {act ? (float)(vw * rd) : 0.f};
      grp.template reduce<4, 1>(s, m);
      rho = m[0];
    };
    double s[4];
    measure(pi, v, w, sl, sh, zl, zh, y, s, rho);
    phi = s[0]; gap = s[1]; dres = s[2]; spent = s[3];
    while (true) {
      // All of these are the same in every thread: uniform exits.
      if (gap <= kGapRel * phi && dres <= fmax(kGapRel * phi, kDualRound * y * budget) &&
          fabs(target - spent) <= kPrimalRel * budget) {
        solved = true;
        break;
      }
      if (steps >= kAllocMaxSteps || !(gap > 0.0) || !(phi <= 1.0e300)) break;
      ++steps;
      const double rp = target - spent, cp = act ? ci * pi : 0.0;
      // Predictor (complementarity target 0) and the cost's solution.
      double rhs[2] = {act ? fma(v, w + bi, -y * cp) : 0.0, cp}, h[2];
      grp.template solve<2>(v, rd, rho, rhs, h);
      double q[2] = {cp * h[0], cp * h[1]};
      grp.template sum<2>(q);
      const double rchc = rcp_newton(q[1]);
      double d = fma(-(q[0] - rp) * rchc, h[1], h[0]) * pi;
      double dl = d * rsl, dh = d * rsh;  // relative steps of the two slacks
      double dzl = -fma(zl, dl, zl), dzh = fma(zh, dh, -zh);
      double t[2] = {act ? (zl - zh) * d : 0.0, act ? (dzl - dzh) * d : 0.0};
      float fl = (float)dl, fh = (float)dh;
      float mx[2] = {act ? fmaxf(-fl, fh) : 0.f, act ? fmaxf(1.f + fl, 1.f - fh) : 0.f};
      grp.template reduce<2, 2>(t, mx);
      const double ap = mx[0] > 1.f ? 1.f / mx[0] : 1.f, az = mx[1] > 1.f ? 1.f / mx[1] : 1.f;
      // sum (z + az dz)(s + ap ds) / gap, with sum s dz = -gap - sum z ds.
      const float q3 =
          (float)((gap + az * (-gap - t[0]) + ap * (t[0] + az * t[1])) * rcp_approx(gap));
      double smu = (double)fminf(fmaxf(q3 * q3 * q3, 1e-6f), 1.f) * (gap * half_inv);
      double d2 = d;
      if (halvings >= 2) {
        d2 *= ap * az;
        if (dres > kGapBehind * gap) smu = fmax(smu, kGapHold * dres * half_inv);
      }
      // Corrector.
      const double tl = (smu - d2 * dzl) * rsl, th = (smu + d2 * dzh) * rsh;
      double rhs1[1] = {act ? fma(tl - th, pi, rhs[0]) : 0.0}, h1[1];
      grp.template solve<1>(v, rd, rho, rhs1, h1);
      double q1[1] = {cp * h1[0]};
      grp.template sum<1>(q1);
      const double dy = (q1[0] - rp) * rchc;
      d = fma(-dy, h[1], h1[0]) * pi;
      dl = d * rsl;
      dh = d * rsh;
      dzl = tl - fma(zl, dl, zl);
      dzh = th + fma(zh, dh, -zh);
      fl = (float)dl;
      fh = (float)dh;
      const float rl = (float)(dzl * rcp_approx(zl)), rh = (float)(dzh * rcp_approx(zh));
      float m1[1] = {act ? fmaxf(fmaxf(-fl, fh), fmaxf(-rl, -rh)) : 0.f};
      double none[1] = {0.0};
      grp.template reduce<1, 1>(none, m1);
      double step = m1[0] > kStepFrac ? kStepFrac / m1[0] : 1.f;
      // The step's point; halved while the residuals grow (they fall in
      // nearly every step: Phi is far from quadratic only near pi_min << 1).
      for (int ls = 0;; ++ls) {
        const double sl2 = fma(step, d, sl), sh2 = fma(-step, d, sh);
        const double zl2 = fma(step, dzl, zl), zh2 = fma(step, dzh, zh), y2 = fma(step, dy, y);
        const double pi2 = act ? (sh2 < sl2 ? 1.0 - sh2 : pmin + sl2) : 1.0;
        const double v2 = rcp_newton(pi2);
        double x[1] = {v2}, r[1];
        grp.template product<1>(x, r);
        float rho2;
        measure(pi2, v2, r[0], sl2, sh2, zl2, zh2, y2, s, rho2);
        if (s[2] + s[1] <= 1.001 * (dres + gap) || s[2] + s[1] <= 1e-11 * s[0] ||
            ls == kAllocMaxBacktrack) {
          sl = sl2; sh = sh2; zl = zl2; zh = zh2; y = y2; pi = pi2; v = v2; w = r[0];
          phi = s[0]; gap = s[1]; dres = s[2]; spent = s[3]; rho = rho2;
          break;
        }
        step *= 0.5;
        if (++halvings == 2) grp.lin = kLinTight;
      }
    }
    if (!solved) status = PAIR_ALLOC_FALLBACK;
  }

  // ---- outputs
  if (!solved && status != PAIR_ALLOC_INVALID) {
    pi = status == PAIR_ALLOC_SLACK ? 1.0
         : (status == PAIR_ALLOC_FLOOR || status == PAIR_ALLOC_INFEASIBLE) ? pmin
                                                                          : budget / sc;
    double x[1] = {1.0 / pi}, r[1];
    grp.template product<1>(x, r);
    double s[2] = {act ? x[0] * (0.5 * r[0] + bi) : 0.0, act ? ci * pi : 0.0};
    grp.template sum<2>(s);
    phi = s[0];
    spent = s[1];
  }
  if (act && sub == 0)
    pi_out[(size_t)g * G + i] =
        status == PAIR_ALLOC_INVALID ? __int_as_float(0x7fc00000) : (float)pi;
  if (threadIdx.x == 0) {
    if (status == PAIR_ALLOC_INVALID) atomicOr(dev_err, PAIR_DEV_ERR_ALLOC_INPUT);
    if (status == PAIR_ALLOC_INFEASIBLE) atomicOr(dev_err, PAIR_DEV_ERR_ALLOC_INFEASIBLE);
    if (stats) {
      double *st = stats + (size_t)g * PAIR_ALLOC_NSTATS;
      st[PAIR_ALLOC_PHI] = phi;
      st[PAIR_ALLOC_SPENT] = spent;
      st[PAIR_ALLOC_GAP] = gap;
      st[PAIR_ALLOC_NEWTON] = (double)steps;
      st[PAIR_ALLOC_STATUS] = (double)status;
    }
  }
}

template <int GP>
pair_status launch_alloc(int32_t B, int32_t G, const float *p_hat, const float *m_hat,
                         const float *a, const float *c_hat, const float *budget, float pi_min,
                         float *pi, double *stats, int32_t *dev_err, cudaStream_t s) {
  const size_t smem =
      sizeof(AllocSmem<GP>) + (size_t)G * alloc_pitch(G) * sizeof(double);
  PAIR_CUDA_TRY(cudaFuncSetAttribute(alloc_kernel<GP>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  PAIR_BEGIN("allocate", s);
  alloc_kernel<GP><<<B, AllocShape<GP>::kThreads, smem, s>>>(G, p_hat, m_hat, a, c_hat, budget,
                                                             pi_min, pi, stats, dev_err);
  PAIR_LAUNCH_CHECK(s);
  return PAIR_OK;
}

}  // namespace
}  // namespace pairk

using namespace pairk;

extern "C" pair_status pair_allocate(int32_t B, int32_t G, const float *p_hat,
                                     const float *m_hat, const float *a, const float *c_hat,
                                     const float *budget, float pi_min, float *pi,
                                     double *stats, int32_t *dev_err, pair_stream_t stream) {
  reset_launches();
  if (B < 1 || G < 2 || G > PAIR_MAX_G || !c_hat || !budget || !pi || !dev_err)
    return PAIR_ERR_INVALID_ARG;
  if (!a && !p_hat) return PAIR_ERR_INVALID_ARG;
  if (!(pi_min > 0.f && pi_min <= 1.f)) return PAIR_ERR_INVALID_ARG;
  const pair_status dv = check_device();
  if (dv != PAIR_OK) return dv;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (G <= 8)
    return launch_alloc<8>(B, G, p_hat, m_hat, a, c_hat, budget, pi_min, pi, stats, dev_err, s);
  if (G <= 16)
    return launch_alloc<16>(B, G, p_hat, m_hat, a, c_hat, budget, pi_min, pi, stats, dev_err, s);
  if (G <= 32)
    return launch_alloc<32>(B, G, p_hat, m_hat, a, c_hat, budget, pi_min, pi, stats, dev_err, s);
  if (G <= 64)
    return launch_alloc<64>(B, G, p_hat, m_hat, a, c_hat, budget, pi_min, pi, stats, dev_err, s);
  return launch_alloc<128>(B, G, p_hat, m_hat, a, c_hat, budget, pi_min, pi, stats, dev_err, s);
}
