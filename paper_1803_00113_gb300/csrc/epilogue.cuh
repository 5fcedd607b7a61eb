// Per-source epilogue (device code shared by the epilogue kernels and the
// per-source Newton step): reduce the per-tile sums of a source, map them from
// each image's natural coordinates to the source's 27 unconstrained
// coordinates, and add the KL term.
//
// Chain rule, exact because every map is applied to reduced sums:
//   per image (affine):  cE_i = calib * kE_i[b], cM_i = calib^2 * kM_i[b],
//                        mu = A u + t, G = A Sigma_s A^T, rho = rho;
//   per source:          kE_i[b] = q_i exp(m_ib + v_ib / 2),
//                        kM_i[b] = q_i exp(2 m_ib + 2 v_ib)     (Sec. 2.1.2,
//                        Eqs. conditional and vareq: E[l|a], E[l^2|a] with
//                        log l ~ N(m, v)),
//                        Sigma_s(angle, radius, axis) = R^T D R (Sec. 2.1.3),
//                        rho = sigmoid(theta_26);
//   grad_theta = J^T grad_nu,
//   hess_theta = J^T H_nu J + sum_a grad_nu[a] * hess_theta(nu_a).
// KL_s follows Eq. kleq, Supplement A and the GMM colour bound of Sec. 4.2.3
// with xi minimised in closed form: -log sum_j w_j exp(-KL(q(c|a) || N_j)).
//
// Precision: the inputs of the chain rule are sums accumulated in FP32 by
// the pixel kernel, so the chain rule and the KL run in FP32 ("real"), which
// adds rounding of the same order as its inputs already carry; the value
// sums (which include the large sky baseline) stay in FP64.  On GB300 an
// FP64 instruction costs ~65 cycles of an SM sub-partition, whatever the
// number of its lanes at work or of independent ones around it.
//
// Bound: latency.  A source is a block of four warps, on the critical path of
// every colour class, and each stage is a short chain of loads, shared
// memory exchanges and barriers.  So the stages that depend on theta alone
// (KL_s, the Jacobian) run beside the reduction of the tile sums, the sums
// come to shared memory in asynchronous copies, maps and indices are formed
// without branches (a divergent 18-way choice of map entries alone took 4k
// cycles a pair), and every small dense product is spread over all threads.
// One source with one 41 x 41 patch per band: 25k cycles (53k before) for
// value, gradient and Hessian; with two 61 x 61 patches per band: 28k (84k).
#pragma once

#include <math.h>

#include <type_traits>

#include "internal.cuh"

namespace celeste {

typedef float real;

constexpr int kNu = 26;   // 20 flux moments (band b, kind e at 4b+e), u (2), Sigma_s (3), rho
constexpr int kNuPad = 32;
constexpr int kKlVals = 8 + 10 + 4;       // per colour component: grad, precision, diag
constexpr int kKlSums = 64;               // per type: mean grad 8, centred outer 36, prec 10, diag 4

static __device__ __forceinline__ real sigm(real t) {
  return t >= 0.f ? 1.f / (1.f + expf(-t)) : expf(t) / (1.f + expf(t));
}
// log(1 + exp(t)) without overflow
static __device__ __forceinline__ real softplus(real t) {
  return t > 0.f ? t + log1pf(expf(-t)) : log1pf(expf(t));
}

constexpr int kEpiThreads = 128;   // four warps per source
constexpr int kPairThreads = kEpiThreads - 32;   // warps 1..3: the pixel sums
constexpr int kPairGroup = 12;                   // pairs reduced between barriers
constexpr int kTileChunk = 32;                   // tiles copied to shared memory at a time

// Barriers among the kPairThreads threads of warps 1..3 (named barrier 1;
// warp 0 is busy with the KL terms meanwhile) and among warps 1 and 2
// (named barrier 2).
static __device__ __forceinline__ void pair_sync() { named_sync(1, kPairThreads); }
static __device__ __forceinline__ void tile_sync() { named_sync(2, 64); }
// Asynchronous copy of 16 bytes to shared memory.
static __device__ __forceinline__ void copy_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}

constexpr int kGeoHess = 55;                     // upper triangle over the 10 w

// The sums of a tile that a pass of this mode has written, kAcc floats apart
// from tile to tile: all of them, or the value and gradient alone; and where
// piece e (16 bytes) of a run of tiles lies, in floats from the first.
template <int kMode>
constexpr int kTileSums = kMode == 2 ? kAcc : kGradAcc;
template <int kMode>
__host__ __device__ constexpr int tile_piece(int e) {
  constexpr int per = kTileSums<kMode> / 4;
  return e / per * kAcc + e % per * 4;
}
static_assert(kAcc % 4 == 0 && kGradAcc % 4 == 0, "whole pieces");

// What a value alone needs of a block's shared memory: half a KB.  (With the
// derivative passes' buffers, 45 KB, five blocks fit on an SM.)
struct KlSmem {
  real th[kNuPad];                 // theta of the source (FP32 copy)
  real kw[kNuPad];                 // colour weights; then grad_nu[a] * kappa_a
  real klj[2 * kMaxColor];         // log w_j - K_j
  real kls[8];                     // scalar KL pieces
  real klt[32];                    // terms of the KL's value and gradient
  double red[2][kEpiThreads / 32]; // per-warp value sums
  double vsum[2];                  // the source's value sums (relative, base)
};

struct EpiSmem : KlSmem {
  float vs[kPairGroup][4];         // per pair of a group: value sums (s, c of relative, base)
  float W[kPairGroup][kAcc];       // per pair of a group: zero, then the other sums (2..63)
  float T[kPairGroup][10 * 10];    // per pair of a group: affine map w <- nu (local)
  alignas(16) float tiles[2][kTileChunk][kAcc];   // tile sums on their way in
  float img[5 * kPairGroup];       // per pair of a group: calibration and A, FP32
  int band[kPairGroup];
  real pw[2 * kKlSums];            // colour bound: pi-weighted sums per type
  real gnu[kNuPad];
  real Hnu[kNu * kNu];
  real J[kNu * kTheta];
  real X[kNu * kTheta + kTheta];   // (padded: read, not used, past the last row)
  real gth[kNuPad];
  real Hth[kTheta * kTheta];
  real DL[20 * kTheta + kTheta];   // d log kappa_a / d theta (padded)
  real D2L[20 * kTheta];           // diagonal second derivatives of log kappa_a
  real kap[kNuPad];                // kappa_a
  real d2S[27];                    // second derivatives of Sigma_s
  real klc[2 * kMaxColor * kKlVals];   // colour-bound pieces per (type, component)
};
template <int kMode>
using EpiShared = std::conditional_t<kMode == 0, KlSmem, EpiSmem>;

// Rows a of J with J[a][c] != 0 for column c: their number and the k-th one
// (the flux coordinates of a type feed every band's kE and kM rows).
static __device__ __forceinline__ int nrows(int c) {
  return c == 0 ? 20 : (c <= 20 ? 10 : (c <= 22 ? 1 : (c <= 25 ? 3 : 1)));
}
// first row and stride of column c's rows
static __device__ __forceinline__ void rows_of(int c, int& r0, int& dr) {
  r0 = c == 0 ? 0 : (c <= 4 ? (c - 1) / 2 : (c <= 20 ? ((c - 5) / 4) & 1 : (c <= 22 ? c - 1 : (c <= 25 ? 22 : 25))));
  dr = c >= 1 && c <= 20 ? 2 : 1;
}

// Row a (0..19) of the flux moments: band b = a / 4, kind e = a % 4 (0: kE0,
// 1: kE1, 2: kM0, 3: kM1): kappa, d log kappa / d theta with its diagonal
// second derivatives, and kappa's row of J.  The eleven coordinates that a
// row depends on are written; the rest of the rows is zero on entry.
static __device__ void kappa_row(const real* th, int a, EpiSmem& S) {
  const int b = a >> 2, e = a & 3;
  const int i = e & 1;
  const bool second = e >= 2;
  const real am = second ? 2.f : 1.f, av = second ? 2.f : 0.5f;
  real* dl = S.DL + a * kTheta;
  real* d2l = S.D2L + a * kTheta;
  real* Ja = S.J + a * kTheta;
  const real q1 = sigm(th[0]), q0 = sigm(-th[0]);
  const real logq = i ? -softplus(-th[0]) : -softplus(th[0]);
  const real l0 = i ? q0 : -q1;
  const int ir = 1 + 2 * i, iv = 2 + 2 * i;
  real m = th[ir], v = expf(th[iv]);
  const real lv = av * v;
  real lm[4], lc[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const real s = colour_select(b, k);
    const real cvk = expf(th[13 + 4 * i + k]);
    m += s * th[5 + 4 * i + k];
    v += s * s * cvk;
    lm[k] = am * s;
    lc[k] = av * s * s * cvk;
  }
  const real kap = expf(logq + am * m + av * v);
  S.kap[a] = kap;
  dl[0] = l0;
  d2l[0] = -q0 * q1;
  Ja[0] = kap * l0;
  dl[ir] = am;
  Ja[ir] = kap * am;
  dl[iv] = d2l[iv] = lv;
  Ja[iv] = kap * lv;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    dl[5 + 4 * i + k] = lm[k];
    Ja[5 + 4 * i + k] = kap * lm[k];
    dl[13 + 4 * i + k] = d2l[13 + 4 * i + k] = lc[k];
    Ja[13 + 4 * i + k] = kap * lc[k];
  }
}

// Derivatives of Sigma_s = (S11, S12, S22) over (angle, log radius, logit axis).
static __device__ void sigma_derivs(const real* th, real dS[3][3], real d2S[3][3][3]) {
  const real phi = th[23], lr = th[24];
  const real ax = sigm(th[25]);
  const real e2 = expf(2.f * lr);
  const real a2 = ax * ax;
  const real a2t = 2.f * a2 * (1.f - ax);
  const real a2tt = 2.f * a2 * (1.f - ax) * (2.f - 3.f * ax);
  const real P = 0.5f * e2 * (1.f + a2), Qd = 0.5f * e2 * (1.f - a2);
  const real Pl = 2.f * P, Pll = 4.f * P, Pt = 0.5f * e2 * a2t, Ptt = 0.5f * e2 * a2tt, Plt = 2.f * Pt;
  const real Ql = 2.f * Qd, Qll = 4.f * Qd, Qt = -0.5f * e2 * a2t, Qtt = -0.5f * e2 * a2tt, Qlt = 2.f * Qt;
  real S2, C2;
  sincosf(2.f * phi, &S2, &C2);
  // S11 = P + Qd C2, S22 = P - Qd C2, S12 = -Qd S2
  for (int e = 0; e < 3; e += 2) {
    const real s = e == 0 ? 1.f : -1.f;
    dS[e][0] = -2.f * s * Qd * S2;
    dS[e][1] = Pl + s * Ql * C2;
    dS[e][2] = Pt + s * Qt * C2;
    d2S[e][0][0] = -4.f * s * Qd * C2;
    d2S[e][0][1] = d2S[e][1][0] = -2.f * s * Ql * S2;
    d2S[e][0][2] = d2S[e][2][0] = -2.f * s * Qt * S2;
    d2S[e][1][1] = Pll + s * Qll * C2;
    d2S[e][1][2] = d2S[e][2][1] = Plt + s * Qlt * C2;
    d2S[e][2][2] = Ptt + s * Qtt * C2;
  }
  dS[1][0] = -2.f * Qd * C2;
  dS[1][1] = -Ql * S2;
  dS[1][2] = -Qt * S2;
  d2S[1][0][0] = 4.f * Qd * S2;
  d2S[1][0][1] = d2S[1][1][0] = -2.f * Ql * C2;
  d2S[1][0][2] = d2S[1][2][0] = -2.f * Qt * C2;
  d2S[1][1][1] = -Qll * S2;
  d2S[1][1][2] = d2S[1][2][1] = -Qlt * S2;
  d2S[1][2][2] = -Qtt * S2;
}

// The terms of KL_s that stand alone, a lane each (lanes 0..8), into S.klt.
template <int kMode>
static __device__ __forceinline__ void kl_lone_terms(const real* th, const ModelDev::F32& f,
                                                     KlSmem& S, int lane) {
  if (lane < 6) {
    // softplus of -+theta_0, -+theta_25, -+theta_26
    const int t = lane < 2 ? 0 : (lane < 4 ? 25 : 26);
    S.klt[lane] = softplus(lane & 1 ? th[t] : -th[t]);
  } else if (lane < 8) {
    const int i = lane - 6;
    const real R1 = f.prior_r[i][0], R2 = f.prior_r[i][1];
    const real rm = th[1 + 2 * i], lrv = th[2 + 2 * i], rv = expf(lrv);
    S.klt[6 + i] =
        0.5f * (f.log_prior_r2[i] - lrv + (rv + (rm - R1) * (rm - R1)) / R2 - 1.f);
    if (kMode >= 1) {
      // gradient of K_i = KL_r + B over the mean and log variance of log r,
      // and its second derivatives
      S.klt[16 + 4 * i] = (rm - R1) / R2;
      S.klt[17 + 4 * i] = 0.5f * (rv / R2 - 1.f);
      S.klt[18 + 4 * i] = 1.f / R2;
      S.klt[19 + 4 * i] = 0.5f * rv / R2;
    }
  } else if (lane == 8) {
    const real lr = th[24], E1 = f.e_radius[0], E2 = f.e_radius[1];
    S.klt[8] = lr + f.half_log_2pi_e2 + (lr - E1) * (lr - E1) / (2.f * E2);
  }
}

// KL_s: value into S.kls[0]; for kMode >= 1 what depends on the type
// probability, radius, axis and profile alone is ADDED (with a minus sign,
// since L = ... - KL) into S.gth and S.Hth, and the rest left in S.pw and
// S.klt for kl_scatter.  By one warp; f and J are the model's FP32 constants
// and its number of colour components.  kApart: warp 2 forms the lone terms
// and meets this warp at named barrier 3.
template <int kMode, bool kApart>
static __device__ void kl_terms(const real* th, const ModelDev::F32& f, int J, EpiShared<kMode>& S,
                                int lane) {
  const real a = sigm(th[0]);
  const real wq = a * (1.f - a);
  if (!kApart) kl_lone_terms<kMode>(th, f, S, lane);
  // ---- colour bound, one lane per (type, component)
  if (lane < 2 * kMaxColor) {
    const int i = lane / kMaxColor, j = lane % kMaxColor;
    if (j < J) {
      const float(*P)[4] = f.color_prec[i][j];
      const real* cm = th + 5 + 4 * i;
      const real* lcv = th + 13 + 4 * i;
      real d[4], cv[4], pd[4];
      real tr = 0.f, quad = 0.f, slv = 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        d[k] = cm[k] - f.color_mean[i][j][k];
        cv[k] = expf(lcv[k]);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        real s = 0.f;
#pragma unroll
        for (int l = 0; l < 4; ++l) s = fmaf(P[k][l], d[l], s);
        pd[k] = s;
        tr = fmaf(P[k][k], cv[k], tr);
        quad = fmaf(d[k], s, quad);
        slv += lcv[k];
      }
      const real K = 0.5f * (tr + quad - 4.f + f.color_logdet[i][j] - slv);
      S.klj[lane] = f.log_color_w[i][j] - K;
      if constexpr (kMode >= 1) {
        real* o = S.klc + lane * kKlVals;
        real gk[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          gk[k] = pd[k];
          gk[4 + k] = 0.5f * (P[k][k] * cv[k] - 1.f);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) o[k] = gk[k];
        int t = 8;
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int l = k; l < 4; ++l) o[t++] = P[k][l];
#pragma unroll
        for (int k = 0; k < 4; ++k) o[t++] = 0.5f * P[k][k] * cv[k];
      }
    } else {
      S.klj[lane] = -INFINITY;
    }
  }
  __syncwarp();
  // ---- per type: softmax weights pi_j = w_j exp(-K_j) / sum (one exp per lane)
  if (lane < 2 * kMaxColor) {
    const int i = lane / kMaxColor;
    real mx = -INFINITY;
#pragma unroll
    for (int j = 0; j < kMaxColor; ++j) mx = fmaxf(mx, S.klj[i * kMaxColor + j]);
    S.kw[lane] = (lane % kMaxColor) < J ? expf(S.klj[lane] - mx) : 0.f;   // scratch
    S.kls[4 + i] = mx;
  }
  __syncwarp();
  real Bval[2], se[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    se[i] = 0.f;
#pragma unroll
    for (int j = 0; j < kMaxColor; ++j) se[i] += S.kw[i * kMaxColor + j];
    Bval[i] = -(S.kls[4 + i] + logf(se[i]));
  }
  if constexpr (kMode >= 1) {
    // pi-weighted sums per type (kKlSums per type): the mean
    // gradient, the precision block and the diagonal ...
    for (int e = lane; e < 2 * kKlVals; e += 32) {
      const int i = e / kKlVals, vv = e % kKlVals;
      real acc = 0.f;
#pragma unroll
      for (int j = 0; j < kMaxColor; ++j)
        if (j < J)
          acc = fmaf(S.kw[i * kMaxColor + j], S.klc[(i * kMaxColor + j) * kKlVals + vv], acc);
      S.pw[i * kKlSums + (vv < 8 ? vv : 36 + vv)] = acc / se[i];
    }
    __syncwarp();
    // ... then the covariance of the gradients across components in centred
    // form, sum_j pi_j (g_j - gbar)(g_j - gbar)^T, which does not cancel
    for (int e = lane; e < (kMode == 2 ? 2 * 36 : 0); e += 32) {
      const int i = e / 36;
      int u = 0, rem = e % 36;
      while (rem >= 8 - u) { rem -= 8 - u; ++u; }
      const int w = u + rem;
      const real gu = S.pw[i * kKlSums + u], gw = S.pw[i * kKlSums + w];
      real acc = 0.f;
#pragma unroll
      for (int j = 0; j < kMaxColor; ++j) {
        const real* gj = S.klc + (i * kMaxColor + j) * kKlVals;
        if (j < J) acc = fmaf(S.kw[i * kMaxColor + j], (gj[u] - gu) * (gj[w] - gw), acc);
      }
      S.pw[i * kKlSums + 8 + (e % 36)] = acc / se[i];
    }
  }
  __syncwarp();
  if (kApart) named_sync(3, 64);
  // ---- value (lane 0)
  if (lane == 0) {
    real v = fmaf(a, (-S.klt[0] - f.log_prior_a), __fmul_rn(1.f - a, (-S.klt[1] - f.log1m_prior_a)));
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const real klr = S.klt[6 + i];
      S.kls[2 + i] = klr + Bval[i];
      v += (i ? a : 1.f - a) * S.kls[2 + i];
    }
    v += S.klt[8];
#pragma unroll
    for (int which = 0; which < 2; ++which) {
      const real b1 = (which ? f.e_profile[0] : f.e_axis[0]);
      const real b2 = (which ? f.e_profile[1] : f.e_axis[1]);
      v += fmaf(b2 - 1.f, S.klt[3 + 2 * which], __fmul_rn(b1 - 1.f, S.klt[2 + 2 * which])) +
           (which ? f.log_beta_profile : f.log_beta_axis);
    }
    S.kls[0] = v;
  }
  __syncwarp();
  if constexpr (kMode >= 1) {
    if (lane == 0) {
      const real la = f.logit_prior_a;
      const real d2q = wq * (1.f - 2.f * a);
      S.gth[0] -= wq * (th[0] - la) + wq * (S.kls[3] - S.kls[2]);
      if (kMode == 2)
        S.Hth[0] -= wq * ((1.f - 2.f * a) * (th[0] - la) + 1.f) + d2q * (S.kls[3] - S.kls[2]);
    } else if (lane == 1) {
      const real lr = th[24], E1 = f.e_radius[0], E2 = f.e_radius[1];
      S.gth[24] -= 1.f + (lr - E1) / E2;
      if (kMode == 2) S.Hth[24 * kTheta + 24] -= 1.f / E2;
    } else if (lane < 4) {
      const int which = lane - 2;
      const int t = which ? 26 : 25;
      const real b1 = (which ? f.e_profile[0] : f.e_axis[0]);
      const real b2 = (which ? f.e_profile[1] : f.e_axis[1]);
      const real sg = sigm(th[t]);
      S.gth[t] -= -(b1 - 1.f) * (1.f - sg) + (b2 - 1.f) * sg;
      if (kMode == 2) S.Hth[t * kTheta + t] -= (b1 + b2 - 2.f) * sg * (1.f - sg);
    }
    __syncwarp();
  }
}

// The rest of the KL's gradient and Hessian, from S.pw and S.klt: the
// blocks of each type's flux coordinates and their products with the type
// probability, an entry a lane.
template <int kMode>
static __device__ __forceinline__ void kl_scatter(const real* th, EpiSmem& S, int lane) {
  const real a = sigm(th[0]);
  const real wq = a * (1.f - a);
  // per type i, local coordinates 0 r-mean, 1 log r-var, 2..5 colour means,
  // 6..9 log colour vars; theta index of local k:
  auto tidx = [](int i, int k) {
    return k == 0 ? 1 + 2 * i : (k == 1 ? 2 + 2 * i : (k < 6 ? 5 + 4 * i + (k - 2) : 13 + 4 * i + (k - 6)));
  };
  // gradient-only mode visits the (i, k, l = 0) entries only
  for (int e0 = lane; e0 < (kMode == 2 ? 200 : 20); e0 += 32) {
    const int e = kMode == 2 ? e0 : (e0 / 10) * 100 + (e0 % 10) * 10;
    const int i = e / 100, k = (e % 100) / 10, l = e % 10;
    const real* pw = S.pw + i * kKlSums;       // grad(8), centred outer(36), prec(10), diag(4)
    real h = 0.f;
    if (k < 2 || l < 2) {
      if (k == l) h = S.klt[18 + 4 * i + k];
    } else {
      const int u = k - 2, w = l - 2;        // colour block 0..7
      const int lo = u < w ? u : w, hi = u < w ? w : u;
      // sum_j pi_j H_j - sum_j pi_j (g_j - gbar)(g_j - gbar)^T
      const int oi = lo * 8 - (lo * (lo - 1)) / 2 + (hi - lo);
      h = -pw[8 + oi];
      if (u < 4 && w < 4) {
        const int po = lo * 4 - (lo * (lo - 1)) / 2 + (hi - lo);
        h += pw[44 + po];
      } else if (u == w) {
        h += pw[54 + (u - 4)];
      }
    }
    const real qi = i ? a : 1.f - a;
    if (kMode == 2) S.Hth[tidx(i, k) * kTheta + tidx(i, l)] -= qi * h;
    if (l == 0) {
      const real dq = i ? wq : -wq;
      const real g = k < 2 ? S.klt[16 + 4 * i + k] : pw[k - 2];
      S.gth[tidx(i, k)] -= qi * g;
      if (kMode == 2) {
        S.Hth[tidx(i, k) * kTheta + 0] -= dq * g;
        S.Hth[0 * kTheta + tidx(i, k)] -= dq * g;
      }
    }
  }
}

// Copies the model's FP32 constants into shared memory (threads tid, tid + n, ...).
static __device__ __forceinline__ void stage_model(ModelDev::F32& dst, const ModelDev* model,
                                                   int tid, int n) {
  constexpr int kWords = sizeof(ModelDev::F32) / 4;
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&model->f);
  uint32_t* d = reinterpret_cast<uint32_t*>(&dst);
  for (int e = tid; e < kWords; e += n) d[e] = src[e];
}

// Slot j of the plan, by the whole block (tid 0..127; S.th holds theta and
// f the model's FP32 constants, in shared memory for kMode >= 1).  kMode: 0 value,
// 1 value + gradient, 2 value + gradient + Hessian.  Warp 0 evaluates the KL
// terms; warps 1 and 2 add up the tile sums, a pair each at a time, while
// warp 3 forms the Jacobian and the images' maps; then the maps are applied
// and the two dense products (X = H_nu J, H_theta += J^T X) formed, an entry
// a thread.  The results are left in S.gth, S.Hth; returns L_rel and L in
// rel and full.
template <int kMode>
static __device__ __forceinline__ void epilogue_source(const PlanView& v,
                                                const ModelDev::F32& f, int n_color,
                                                EpiShared<kMode>& S, int j, int tid, bool pixel_only,
                                                double& rel, double& full) {
  const int lane = tid & 31, wid = tid >> 5;
  const real* th = S.th;
  const int p0 = v.slot_pair_ptr[j], p1 = v.slot_pair_ptr[j + 1];
  if constexpr (kMode >= 1) {
    if (tid < kNuPad) S.gnu[tid] = S.gth[tid] = 0.f;
    for (int e = tid; e < kNu * kTheta; e += kEpiThreads) S.J[e] = 0.f;
    for (int e = tid; e < 20 * kTheta; e += kEpiThreads) S.DL[e] = S.D2L[e] = 0.f;
  }
  if constexpr (kMode == 2) {
    for (int e = tid; e < kNu * kNu; e += kEpiThreads) S.Hnu[e] = 0.f;
    for (int e = tid; e < kTheta * kTheta; e += kEpiThreads) S.Hth[e] = 0.f;
  }
  __syncthreads();
  if (wid == 0) {
    if (!pixel_only) {
      kl_terms<kMode, (kMode >= 1)>(th, f, n_color, S, lane);
      if constexpr (kMode >= 1) kl_scatter<kMode>(th, S, lane);
    }
  } else {
    const int u = tid - 32;                            // 0 .. kPairThreads - 1
    double vr = 0.0, vb = 0.0;
    if constexpr (kMode == 0) {
      // value sums of every pair's items, thread-strided, then one reduction;
      // with three pairs or more of up to an item a thread, eight pairs' items
      // are loaded together (one or two pairs, or longer ones, lose 0.6-1 us of
      // 9-22 that way)
      for (int pg = p0; pg < p1; pg += 8) {
        int ib[8], ie[8], most = 0;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          ib[g] = ie[g] = 0;
          if (pg + g < p1) {
            ib[g] = v.pairs[pg + g].item_begin;
            ie[g] = v.pairs[pg + g].item_end;
          }
          most = max(most, ie[g] - ib[g]);
        }
        if (p1 - pg < 3 || most > kPairThreads) {
          for (int pp = pg; pp < min(pg + 8, p1); ++pp) {
            const int b = v.pairs[pp].item_begin, e = v.pairs[pp].item_end;
            for (int it = b + u; it < e; it += kPairThreads) {
              vr += (double)v.vpartials[2 * (size_t)it];
              vb += (double)v.vpartials[2 * (size_t)it + 1];
            }
          }
          continue;
        }
        float2 x[8];
#pragma unroll
        for (int g = 0; g < 8; ++g)
          if (ib[g] + u < ie[g]) x[g] = reinterpret_cast<const float2*>(v.vpartials)[ib[g] + u];
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          if (ib[g] + u < ie[g]) {
            vr += (double)x[g].x;
            vb += (double)x[g].y;
          }
        }
      }
      vr = warp_sum_d(vr);
      vb = warp_sum_d(vb);
      if (lane == 0) {
        S.red[0][wid - 1] = vr;
        S.red[1][wid - 1] = vb;
      }
      pair_sync();
      if (u == 0) {
        S.vsum[0] = S.red[0][0] + S.red[0][1] + S.red[0][2];
        S.vsum[1] = S.red[1][0] + S.red[1][1] + S.red[1][2];
      }
    } else {
      // thread u's entry of H_nu (upper triangle of the ten w, u < 55) or of
      // grad_nu (the next ten): the terms of its sum over the w, as offsets
      // into T and W; terms it does not have multiply entry 0 of W, zero
      auto lo = [](int a) { return a < 4 ? a : (a < 6 ? 4 : (a < 9 ? 6 : 9)); };
      auto hi = [](int a) { return a < 4 ? a + 1 : (a < 6 ? 6 : (a < 9 ? 9 : 10)); };
      const bool ghess = u < kGeoHess, ggrad = u >= kGeoHess && u < kGeoHess + kW;
      int ea = ghess ? 0 : min(u - kGeoHess, kW - 1), ec = ea;
      int tk[3], tl[3], wo[9];
      if (ghess) {
        int r = u;
        while (r >= 10 - ea) { r -= 10 - ea; ++ea; }
        ec = ea + r;
      }
      const int ka = lo(ea), la = lo(ec), na3 = hi(ea) - ka, nc3 = ghess ? hi(ec) - la : 1;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        tk[i] = i < na3 ? (ka + i) * 10 + ea : 99;
        tl[i] = ghess && i < nc3 ? (la + i) * 10 + ec : 99;
      }
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const int k = ka + q / 3, l = la + q % 3, kk = min(k, l), ll = max(k, l);
        const bool zero = ghess && kk >= 2 && kk <= 3 && ll <= 3;   // (cM, cM): vanish
        const bool on = q / 3 < na3 && q % 3 < nc3 && !zero;
        wo[q] = !on ? 0 : (ghess ? hidx(kk, ll) : 2 + k);
      }
      // what depends on theta alone, while the first loads are on their way:
      // the KL's lone terms (warp 2), the geometric rows of J (warp 1) and its
      // flux rows (warp 3)
      auto apart = [&] {
        if (wid == 2) {
          kl_lone_terms<kMode>(th, f, S, lane);
          named_arrive(3, 64);
        } else if (wid == 3) {
          if (lane < 20) kappa_row(th, lane, S);
        } else if (lane == 0) {
          real dS[3][3], d2S[3][3][3];
          sigma_derivs(th, dS, d2S);
#pragma unroll
          for (int e = 0; e < 3; ++e)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              S.J[(22 + e) * kTheta + 23 + c] = dS[e][c];
#pragma unroll
              for (int d = 0; d < 3; ++d) S.d2S[9 * e + 3 * c + d] = d2S[e][c][d];
            }
          S.J[20 * kTheta + 21] = S.J[21 * kTheta + 22] = 1.f;
          const real r = sigm(th[26]);
          S.J[25 * kTheta + 26] = r * (1.f - r);
        }
        __syncwarp();
      };
      if (p0 == p1) apart();
      for (int pp = p0; pp < p1; pp += kPairGroup) {
        const int ng = min(kPairGroup, p1 - pp);
        int ib = 0, ie = 0, im = 0;
        if (lane < ng) {
          const PairInfo& pi = v.pairs[pp + lane];
          ib = pi.item_begin;
          ie = pi.item_end;
          im = pi.image;
          if (wid == 3) S.band[lane] = pi.band;
        }
        if (wid < 3) {
          // the tile sums of the group's pairs, whose items are contiguous:
          // chunks of kTileChunk tiles (256 B each; 48 B without a Hessian) are
          // copied to shared memory, one chunk ahead, and warps 1 and 2 add up
          // a pair each at a time: lane l forms accumulators 2 l and 2 l + 1 by
          // compensated (Kahan) FP32 summation in tile order, whose error does
          // not grow with the number of tiles
          const int t0 = __shfl_sync(0xffffffffu, ib, 0);
          const int t1 = __shfl_sync(0xffffffffu, ie, ng - 1);
          auto fetch = [&](int c) {
            const int n16 = min(kTileChunk, t1 - t0 - c * kTileChunk) * (kTileSums<kMode> / 4);
            const float* src = v.partials + (size_t)(t0 + c * kTileChunk) * kAcc;
            float* dst = &S.tiles[c & 1][0][0];
            for (int e = u; e < n16; e += 64)
              copy_async16(dst + tile_piece<kMode>(e), src + tile_piece<kMode>(e));
            asm volatile("cp.async.commit_group;" ::: "memory");
          };
          const int nc = (t1 - t0 + kTileChunk - 1) / kTileChunk;
          fetch(0);
          if (pp == p0) apart();
          int g = wid - 1;
          float2 s = make_float2(0.f, 0.f), c = s;
          for (int ch = 0; ch < nc; ++ch) {
            if (ch + 1 < nc) {
              fetch(ch + 1);
              asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
              asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            tile_sync();
            const int c0 = t0 + ch * kTileChunk, c1 = c0 + kTileChunk;
            const float2* x = reinterpret_cast<const float2*>(&S.tiles[ch & 1][0][0]) + lane;
            while (g < ng) {
              const int b = __shfl_sync(0xffffffffu, ib, g), e = __shfl_sync(0xffffffffu, ie, g);
              if (b >= c1) break;
              const int q1 = 2 * lane < kTileSums<kMode> ? min(e, c1) - c0 : 0;
#pragma unroll 4
              for (int q = max(b, c0) - c0; q < q1; ++q) {
                const float2 y = x[q * (kAcc / 2)];
                const float ya = y.x - c.x, yb = y.y - c.y;
                const float ta = s.x + ya, tb = s.y + yb;
                c.x = (ta - s.x) - ya;
                c.y = (tb - s.y) - yb;
                s.x = ta;
                s.y = tb;
              }
              if (e > c1) break;                       // goes on in the next chunk
              // the value sums go on in FP64; the others are used in FP32,
              // and s - c rounded once to FP32 equals (float)((double)s -
              // (double)c): that double difference is exact or off s by far
              // less than half an FP32 unit in the last place
              if (lane == 0) {
                S.W[g][0] = 0.f;
                S.vs[g][0] = s.x;
                S.vs[g][1] = c.x;
                S.vs[g][2] = s.y;
                S.vs[g][3] = c.y;
              } else if (2 * lane < kTileSums<kMode>) {
                S.W[g][2 * lane] = s.x - c.x;
                S.W[g][2 * lane + 1] = s.y - c.y;
              }
              s = c = make_float2(0.f, 0.f);
              g += 2;
            }
            tile_sync();                               // before the buffer is filled again
          }
        } else {
          // each pair's local affine map, FP32: w_k = sum_a T[k][a] nu_a;
          // five values of an image (calibration, A) in five lanes, so that
          // six images share a conversion; then an entry (of the eighteen that
          // are not zero) of a pair a lane, from two of the values (three bits
          // an entry in kOne, kTwo): kind 0 the first, 1 the product, 2 twice
          // it, 3 A0 A3 + A1 A2, 4 one
          static_assert(kPairGroup == 12, "two conversions");
          double raw[2];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int q = lane % 5;
            const int image = __shfl_sync(0xffffffffu, im, min(6 * c + min(lane / 5, 5), ng - 1));
            const celeste_image& I = v.images[image];
            raw[c] = q == 0 ? I.calib : I.wcs_A[q - 1];
          }
          if (pp == p0) apart();
#pragma unroll
          for (int c = 0; c < 2; ++c)
            if (lane < 30) S.img[30 * c + lane] = (float)raw[c];
          __syncwarp();
          constexpr uint64_t kKind = 0412113112100001100ull, kOne = 043321121143210000ull,
                             kTwo = 044344322100000000ull;
          for (int q = lane; q < 18 * ng; q += 32) {
            const int g = q / 18, e = q - 18 * g, sh = 3 * e;
            const int kind = (int)(kKind >> sh & 7);
            const float* I = S.img + 5 * g;
            const float f1 = I[kOne >> sh & 7], f2 = I[kTwo >> sh & 7], f3 = I[2], f4 = I[3];
            const float t = kind == 0 ? f1
                                      : (kind == 1 ? f1 * f2
                                                   : (kind == 2 ? 2.f * f1 * f2
                                                                : (kind == 3 ? fmaf(f3, f4, __fmul_rn(f1, f2)) : 1.f)));
            const int te = e < 4 ? 11 * e
                                 : (e < 8 ? 44 + ((e - 4) >> 1) * 10 + (e & 1)
                                          : (e < 17 ? 66 + (e - 8) / 3 * 10 + (e - 8) % 3 : 99));
            S.T[g][te] = t;
          }
        }
        pair_sync();
        // the maps applied, in pair order, an entry a thread
        if ((kMode == 2 && ghess) || ggrad) {
          for (int g = 0; g < ng; ++g) {
            const float* T = S.T[g];
            const float* W = S.W[g];
            const int b = S.band[g];
            float x[9], p[9], val = 0.f;
#pragma unroll
            for (int q = 0; q < 9; ++q) {
              x[q] = W[wo[q]];
              p[q] = T[tk[q / 3]] * T[tl[q % 3]];    // (entry 99 of T is one)
            }
#pragma unroll
            for (int q = 0; q < 9; ++q) val = fmaf(p[q], x[q], val);
            const int na = ea < 4 ? 4 * b + ea : 16 + ea, nc = ec < 4 ? 4 * b + ec : 16 + ec;
            if (ghess) S.Hnu[na * kNu + nc] += val;
            else S.gnu[na] += val;                   // nu of w_a (4..9 -> 20..25)
          }
        }
        if (wid == 1) {
          // the value sums of the group's pairs, in pair order: lane 2 g + h
          // holds pair g's relative (h = 0) or base sum, lanes 0 and 1 add
          double d = 0.0;
          if (lane < 2 * ng) {
            const float* x = S.vs[lane >> 1] + 2 * (lane & 1);
            d = (double)x[0] - (double)x[1];
          }
          for (int g = 0; g < ng; ++g) vr += __shfl_sync(0xffffffffu, d, 2 * g + (lane & 1));
        }
        if (pp + kPairGroup < p1) pair_sync();
      }
      // the lower triangle of H_nu, by the threads that formed the upper one
      if (kMode == 2 && ghess && ea != ec) {
        if (ea >= 4) {
          S.Hnu[(16 + ec) * kNu + 16 + ea] = S.Hnu[(16 + ea) * kNu + 16 + ec];
        } else {
#pragma unroll
          for (int b = 0; b < 5; ++b) {
            const int na = 4 * b + ea, nc = ec < 4 ? 4 * b + ec : 16 + ec;
            S.Hnu[nc * kNu + na] = S.Hnu[na * kNu + nc];
          }
        }
      }
      if (wid == 1 && lane < 2) S.vsum[lane] = vr;
    }
  }
  __syncthreads();
  const double kl = pixel_only ? 0.0 : (double)S.kls[0];
  rel = S.vsum[0] - kl;
  full = S.vsum[1] + S.vsum[0] - kl;
  if constexpr (kMode >= 1) {
    if constexpr (kMode == 2) {
      if (tid < 20) S.kw[tid] = S.gnu[tid] * S.kap[tid];
      __syncthreads();
      // X = H_nu J where J's column has support.  Columns 0..20 (ten or
      // twenty rows): thread (c, g) forms rows a = g, g + 4, ... of column c,
      // seven chains sharing each entry of J; the other columns (one or three
      // rows), an entry a thread
      if (tid < 4 * 21) {
        const int c = tid % 21, g = tid / 21, nr = nrows(c);
        int r, dr;
        rows_of(c, r, dr);
        real x[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 5
        for (int k = 0; k < nr; ++k, r += dr) {
          const real jv = S.J[r * kTheta + c];
#pragma unroll
          for (int m = 0; m < 7; ++m)
            x[m] = fmaf(S.Hnu[min(g + 4 * m, kNu - 1) * kNu + r], jv, x[m]);
        }
#pragma unroll
        for (int m = 0; m < 7; ++m)
          if (g + 4 * m < kNu) S.X[(g + 4 * m) * kTheta + c] = x[m];
      } else {
        for (int e = tid - 4 * 21; e < 6 * kNu; e += kEpiThreads - 4 * 21) {
          const int c = 21 + e % 6, a = e / 6, nr = nrows(c);
          int r, dr;
          rows_of(c, r, dr);
          real x = 0.f;
          for (int k = 0; k < nr; ++k) x = fmaf(S.Hnu[a * kNu + r + k], S.J[(r + k) * kTheta + c], x);
          S.X[a * kTheta + c] = x;
        }
      }
      if (tid < 9) {
        // Sigma_s second-order chain term
        real h = 0.f;
#pragma unroll
        for (int e = 0; e < 3; ++e) h += S.gnu[22 + e] * S.d2S[9 * e + tid];
        S.Hth[(23 + tid / 3) * kTheta + 23 + tid % 3] += h;
      } else if (tid == 32) {
        const real r = sigm(th[26]);
        S.Hth[26 * kTheta + 26] += S.gnu[25] * r * (1.f - r) * (1.f - 2.f * r);
      }
    }
    __syncthreads();
    // gradient: J^T grad_nu over each column's rows
    if (tid >= kEpiThreads - kTheta) {
      const int c = tid - (kEpiThreads - kTheta), nr = nrows(c);
      int r, dr;
      rows_of(c, r, dr);
      real gsum = 0.f;
#pragma unroll 5
      for (int k = 0; k < nr; ++k, r += dr) gsum = fmaf(S.J[r * kTheta + c], S.gnu[r], gsum);
      S.gth[c] += gsum;
    }
    if constexpr (kMode == 2) {
      // Hth += J^T X over d >= c (mirrored), plus the flux-moment
      // second-order term sum_a kw_a (dl dl^T + diag d2l).  Column 0 (twenty
      // rows) has a thread for each d; thread (c, g) of the others takes d =
      // c + g, c + g + 3, ..., nine chains sharing the entries of column c.
      auto entry = [&](int c, int d, real x) {
        S.Hth[c * kTheta + d] += x;
        if (d != c) S.Hth[d * kTheta + c] += x;
      };
      if (tid < kTheta) {
        const int d = tid;
        real x = 0.f;
#pragma unroll 10
        for (int r = 0; r < 20; ++r) x = fmaf(S.J[r * kTheta], S.X[r * kTheta + d], x);
        if (d <= 20) {
#pragma unroll 10
          for (int r = 0; r < 20; ++r) {
            const real kd = S.kw[r] * S.DL[r * kTheta];
            x = fmaf(kd, S.DL[r * kTheta + d], x);
            if (d == 0) x = fmaf(S.kw[r], S.D2L[r * kTheta], x);
          }
        }
        entry(0, d, x);
      } else if (tid < kTheta + 3 * (kTheta - 1)) {
        constexpr int kCh = 9;
        const int c = 1 + (tid - kTheta) % (kTheta - 1), g = (tid - kTheta) / (kTheta - 1);
        const int nr = nrows(c);
        int r0, dr;
        rows_of(c, r0, dr);
        const int step = dr * kTheta;
        real x[kCh];
#pragma unroll
        for (int m = 0; m < kCh; ++m) x[m] = 0.f;
        // (chains with d past the last column run on what follows and are
        // dropped; DL's columns beyond 20 are zero)
        const real* Jc = S.J + r0 * kTheta + c;
        const real* Xd = S.X + r0 * kTheta + c + g;
#pragma unroll 2
        for (int k = 0; k < nr; ++k, Jc += step, Xd += step) {
          const real jv = *Jc;
#pragma unroll
          for (int m = 0; m < kCh; ++m) x[m] = fmaf(jv, Xd[3 * m], x[m]);
        }
        if (c <= 20) {
          const real* kw = S.kw + r0;
          const real* Lc = S.DL + r0 * kTheta + c;
          const real* L2 = S.D2L + r0 * kTheta + c;
#pragma unroll 2
          for (int k = 0; k < nr; ++k, kw += dr, Lc += step, L2 += step) {
            const real kd = *kw * *Lc;
#pragma unroll
            for (int m = 0; m < kCh; ++m) x[m] = fmaf(kd, Lc[g + 3 * m], x[m]);
            if (g == 0) x[0] = fmaf(*kw, *L2, x[0]);
          }
        }
#pragma unroll
        for (int m = 0; m < kCh; ++m)
          if (c + g + 3 * m < kTheta) entry(c, c + g + 3 * m, x[m]);
      }
    }
    __syncthreads();
  }
}

}  // namespace celeste
