// Per-(source, image) setup of one pair, by one warp: the PSF-convolved
// Gaussian components of the star and galaxy light kernels in the patch's
// pixel frame, and the flux moments of each source type in the image's band,
// as an FP32 record (positions relative to the patch origin so that FP32
// keeps them exact to ~1e-6 px).
//
// Follows Sec. 2.1.2 (flux: l_b = r exp(S_b . c), log-normal r and normal
// colours under q), Sec. 2.1.3 (Eq. eq:hsi and Sigma_s = R^T D R), Sec. 2.2
// (calibration, linear WCS, Gaussian-mixture PSF) and the Gaussian-Gaussian
// convolution of Sec. 2.2.3.
//
// Included by the translation units whose kernels form records: the setup
// kernel itself, the per-class preparation kernel and the per-source step.
#pragma once

#include <math.h>

#include "internal.cuh"

namespace celeste {

__device__ __forceinline__ float sigmoid_f(float t) {
  return t >= 0.f ? 1.f / (1.f + expf(-t)) : expf(t) / (1.f + expf(t));
}

// Record of pair p, by the calling warp (lanes over Gaussian components).
// Only the patch-local centre needs FP64 (reference-frame positions reach
// ~2000 px); everything else is FP32, which keeps the records exact to ~1e-7
// relative.  On this GPU the FP64 pipe also carries the double -> float
// conversions, at about one warp instruction per 64 cycles of an SM
// sub-partition, so the warp converts its theta row and its image's PSF,
// WCS and calibration with one instruction each (a value per lane), shared
// through thf and imf: 32 floats each of the warp's shared memory; the centre's
// two coordinates and the flux moments' two types are formed side by side, in
// even and odd lanes.  image, x0, y0: the pair's; th: its source's theta.
__device__ __forceinline__ void setup_pair(const PlanView& v, const ModelDev* __restrict__ model,
                                           int p, int image, int x0, int y0, const double* th,
                                           float* thf, float* imf, int lane) {
  const celeste_image& im = v.images[image];
  float* rec = v.records + (size_t)p * kRecF;
  constexpr int kPsfV = 6 * kPsf;                // PSF values: weight, mean (2), covariance (3)
  static_assert(kTheta <= 32 && kPsfV + 5 <= 32, "one value per lane");
  __syncwarp();
  float tv;                                      // this lane's theta
  {
    const double* src = lane < kPsfV ? &im.psf[0][0] + lane
                                     : (lane < kPsfV + 4 ? im.wcs_A + (lane - kPsfV) : &im.calib);
    const double t = th[lane < kTheta ? lane : 0], i = *src;
    thf[lane] = tv = (float)t;
    imf[lane] = (float)i;
  }
  __syncwarp();
  const float* psf = imf;                        // psf[6 k + c]
  const float* wcs = imf + kPsfV;                // A0, A1, A2, A3, calib

  // centre in the patch's local pixel frame (FP64, then FP32): x in the even
  // lanes, y in the odd ones
  const int odd = lane & 1;
  const double ux = th[21], uy = th[22];
  const float mul = (float)(im.wcs_A[2 * odd] * ux + im.wcs_A[2 * odd + 1] * uy + im.wcs_t[odd] -
                            (double)(odd ? y0 : x0));
  const float mux = __shfl_sync(0xffffffffu, mul, 0), muy = __shfl_sync(0xffffffffu, mul, 1);
  // Sigma_s = R^T diag(d1, d2) R, R = [[c, -s], [s, c]]  (Sec. 2.1.3)
  float s, c;
  sincosf(thf[23], &s, &c);
  const float rad2 = expf(2.f * thf[24]);
  const float axis = sigmoid_f(thf[25]);
  const float d1 = rad2, d2 = axis * axis * rad2;
  const float S11 = c * c * d1 + s * s * d2;
  const float S12 = c * s * (d2 - d1);
  const float S22 = s * s * d1 + c * c * d2;
  // G = A Sigma_s A^T
  const float a11 = wcs[0], a12 = wcs[1];
  const float a21 = wcs[2], a22 = wcs[3];
  const float t11 = a11 * S11 + a12 * S12, t12 = a11 * S12 + a12 * S22;
  const float t21 = a21 * S11 + a22 * S12, t22 = a21 * S12 + a22 * S22;
  const float g11 = t11 * a11 + t12 * a12;
  const float g12 = t11 * a21 + t12 * a22;
  const float g22 = t21 * a21 + t22 * a22;

  const int ne = model->n_exp, nd = model->n_dev;
  const int ncomp = kPsf * (1 + ne + nd);
  const float log2_2pi = 2.6514961294723187f;   // log2(2 pi)
  for (int ci = lane; ci < ncomp; ci += 32) {
    int k;
    float tau, weight;
    if (ci < kPsf) {
      k = ci;
      tau = 0.f;
      weight = psf[6 * k];
    } else {
      const int r = ci - kPsf;
      k = r / (ne + nd);
      const int j = r % (ne + nd);
      // the weight product stays FP64 (one rounding), as the oracle's
      if (j < ne) {
        tau = model->f.tau_exp[j];
        weight = (float)(im.psf[k][0] * model->alpha_exp[j]);
      } else {
        tau = model->f.tau_dev[j - ne];
        weight = (float)(im.psf[k][0] * model->alpha_dev[j - ne]);
      }
    }
    const float cxx = fmaf(tau, g11, psf[6 * k + 3]);
    const float cxy = fmaf(tau, g12, psf[6 * k + 4]);
    const float cyy = fmaf(tau, g22, psf[6 * k + 5]);
    const float det = cxx * cyy - cxy * cxy;
    const float rdet = 1.f / det;
    float* e = rec + kHdr + ci * kCompF;
    e[C_MX] = mux + psf[6 * k + 1];
    e[C_MY] = muy + psf[6 * k + 2];
    e[C_P11] = cyy * rdet;
    e[C_P12] = -cxy * rdet;
    e[C_P22] = cxx * rdet;
    e[C_LW] = log2f(weight) - log2_2pi - 0.5f * log2f(det);
    e[C_TAU] = tau;
    e[7] = 0.f;
  }

  // flux moments per type in this image's band (Sec. 2.1.2), a type a lane;
  // the exponentials of the log variances first, a coordinate a lane
  const float ex = expf(tv);
  const int b = im.band, i = lane & 1;
  float m = thf[1 + 2 * i];
  float var = __shfl_sync(0xffffffffu, ex, 2 + 2 * i);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float sel = colour_select(b, q);
    m += sel * thf[5 + 4 * i + q];
    var += sel * sel * __shfl_sync(0xffffffffu, ex, 13 + 4 * i + q);
  }
  if (lane < 2) {
    const float kk = wcs[4] * expf(m + 0.5f * var);   // calib E[l_b | a=i]
    const float ev = expm1f(var);                       // E[l^2] / E[l]^2 - 1
    const float qi = sigmoid_f(i ? thf[0] : -thf[0]);
    rec[H_CE0 + i] = qi * kk;
    rec[H_CM0 + i] = qi * kk * kk * (1.f + ev);
    rec[H_K0 + i] = kk;
    rec[H_EV0 + i] = ev;
    rec[H_Q0 + i] = qi;
    rec[H_RHO + i] = sigmoid_f(i ? -thf[26] : thf[26]);
    rec[12 + i] = rec[14 + i] = 0.f;
  }
}

__device__ __forceinline__ void setup_pair(const PlanView& v, const ModelDev* __restrict__ model,
                                           int p, bool use_trial, float* thf, float* imf,
                                           int lane) {
  const PairInfo& pi = v.pairs[p];
  const double* th = use_trial && pi.slot >= 0 ? v.theta_trial + (size_t)pi.slot * kTheta
                                               : v.theta + (size_t)pi.source * kTheta;
  setup_pair(v, model, p, pi.image, pi.x0, pi.y0, th, thf, imf, lane);
}

}  // namespace celeste
