// Pixel kernels: the hot loop of the method.
//
// For every (source, image patch, pixel tile) work item, one warp stages the
// pair's component record in shared memory and each lane walks its pixels:
//   * renders the source's galaxy and star profile densities with their
//     first and second derivatives in the image's natural coordinates
//     (centre mu, shape G = A Sigma_s A^T, profile weight rho) -- Sec. 2.2.3;
//   * forms E = bgE + E_s and V = bgV + V_s (Eqs. conditional, vareq) and the
//     delta-method pixel term -E + x (log E - V / (2 E^2)) (Eq. eq:log_p_last,
//     Sec. 4.2.2) with its partials;
//   * accumulates the value, the gradient and the Hessian over the 10
//     per-image natural coordinates w = (cE0, cE1, cM0, cM1, mu, G, rho).
// The 64 sums are reduced over the lanes (the two value sums by shuffles, the
// others along their rows of a tile in shared memory; the gradient kernel's
// twelve by shuffles) and written to the item's slot; the epilogue adds a
// pair's items (compensated FP32, the value sums in FP64) and chains them to
// the 27 coordinates.
//
// Derivatives of a Gaussian component with respect to its covariance come
// from the heat equation (d phi / dC_ab = 1/2 d^2 phi / dmu_a dmu_b), so the
// kernel only needs the Hermite polynomials of orders 0..4 in y = P (p - mu).
#include <math.h>

#include <type_traits>

#include "device_once.h"
#include "internal.cuh"
#include "launch_rules.h"
#include "overlap.h"
#include "setup.cuh"

namespace celeste {

constexpr float kHalfLog2e = 0.72134752044448170368f;   // log2(e) / 2

// ---- staged records
// Every pixel kernel stages the (source, image) record of its work item in
// the warp's shared memory, built from the global record (8 floats per
// component: mx, my, P11, P12, P22, lw, tau) in one of two layouts:
//   value layout:  header | origins | star {A11, A12, A22, lw}
//                                   | per PSF component k: galaxy pairs, then singles
//   derivs layout: header | origins | star {A, lw | P, 0}
//                                   | per PSF component k: galaxy pairs, then singles
// (with the pairs' skip radii between origins and stars, see stage_skip).
// A galaxy component has 20 values {A, lw | -P11, -P12, -P22, tau |
// -2 P12, -2 P11^2, -2 P22^2, -2 P12^2 | -4 P12, -2 P12 P11, -2 P12 P22,
// -2 P11 | -2 P22, -4 P11, -4 P22, 0}: the signs are chosen so that no
// formula below negates an operand.  An FP32 instruction with three distinct
// register operands issues every 3 cycles per 64 lanes here (1.55 per 32),
// with two every 2, so sums with a constant multiple of P take it staged, as
// an addition, rather than as an FMA with 2 or 4.  The components of PSF
// component k come in pairs (exponential j, de Vaucouleurs j) for
// j < min(n_exp, n_dev), their values interleaved (exponential in the even
// slots), so that one packed two-wide FP32 instruction (ffma2, which rounds
// each half as fmaf does) evaluates both; the components without a partner
// follow with their 20 values in a row.
// A = -log2(e)/2 (P11, 2 P12, P22) are the coefficients of the exponent's
// quadratic form: log2 phi = lw + A11 dx^2 + A12 dx dy + A22 dy^2.  Every
// component convolved with PSF component k has that component's mean (the
// source centre plus the PSF offset), so a kernel forms the pixel's offset
// and its products once per k from the "origins".  Both layouts evaluate
// phi with the same instructions: a value-only kernel and the derivative
// kernel give bit-identical densities for the same record.
constexpr int kOrgF = 8;                                   // (mx, my) per k, padded
constexpr int kValF = 4;
constexpr int kStarF = 8;
constexpr int kGalF = 20;
constexpr int kSkipBase = kHdr + kOrgF;                    // skip radii, kMaxProf per k
constexpr int kCompBase = kSkipBase + kPsf * kMaxProf;
constexpr int kValRecF = kCompBase + kMaxComp * kValF;
constexpr int kDerivRecF = kCompBase + kPsf * kStarF + kPsf * 2 * kMaxProf * kGalF;
static_assert(2 * kPsf <= kOrgF && kValRecF % 4 == 0 && kDerivRecF % 4 == 0, "staged layout");

__device__ __forceinline__ float4 quad_coeffs(float p11, float p12, float p22, float lw) {
  return make_float4(-kHalfLog2e * p11, (-2.f * kHalfLog2e) * p12, -kHalfLog2e * p22, lw);
}

// Stages the record at src (global) into dst (the warp's shared memory);
// n_comp = kPsf (1 + n_exp + n_dev) components in the global order (stars,
// then per PSF component the exponential and de Vaucouleurs components).
template <bool kDerivs>
__device__ __forceinline__ void stage_record(float* __restrict__ dst, const float* __restrict__ src,
                                             int n_comp, int lane, int n_exp = 0) {
  const float4* s4 = reinterpret_cast<const float4*>(src);
  float4* d4 = reinterpret_cast<float4*>(dst);
  if (lane < kHdr / 4) d4[lane] = s4[lane];
  if (lane < kPsf)
    *reinterpret_cast<float2*>(dst + kHdr + 2 * lane) =
        *reinterpret_cast<const float2*>(src + kHdr + lane * kCompF);
  for (int ci = lane; ci < n_comp; ci += 32) {
    const float4 a = s4[kHdr / 4 + 2 * ci];
    const float4 b = s4[kHdr / 4 + 2 * ci + 1];
    const float p11 = a.z, p12 = a.w, p22 = b.x;
    const float4 q = quad_coeffs(p11, p12, p22, b.y);
    if (!kDerivs) {
      if (ci < kPsf) {
        d4[kCompBase / 4 + ci] = q;
      } else {
        // galaxy: pairs (exponential j, de Vaucouleurs j) interleaved, then
        // the components without a partner
        const int per = (n_comp - kPsf) / kPsf;
        const int g = ci - kPsf, k = g / per, jj = g - k * per;
        const int nb = n_exp < per - n_exp ? n_exp : per - n_exp;
        const bool dev = jj >= n_exp;
        const int j = dev ? jj - n_exp : jj;
        float* base = dst + kCompBase + (kPsf + k * per) * kValF;
        if (j < nb) {
          float* o = base + j * 2 * kValF + (dev ? 1 : 0);
          o[0] = q.x;
          o[2] = q.y;
          o[4] = q.z;
          o[6] = q.w;
        } else {
          const int single = dev ? (n_exp - nb) + (j - nb) : j - nb;
          *reinterpret_cast<float4*>(base + nb * 2 * kValF + single * kValF) = q;
        }
      }
    } else if (ci < kPsf) {
      float4* o = reinterpret_cast<float4*>(dst + kCompBase + ci * kStarF);
      o[0] = q;
      o[1] = make_float4(p11, p12, p22, 0.f);
    } else {
      // galaxy component: PSF component k, index j of its profile
      const int per = (n_comp - kPsf) / kPsf;
      const int g = ci - kPsf, k = g / per, jj = g - k * per;
      const int ne = n_exp;
      const int nb = ne < per - ne ? ne : per - ne;
      const bool dev = jj >= ne;
      const int j = dev ? jj - ne : jj;
      const float vals[kGalF] = {q.x, q.y, q.z, q.w, -p11, -p12, -p22, b.z,
                                 -2.f * p12, -2.f * p11 * p11, -2.f * p22 * p22, -2.f * p12 * p12,
                                 -4.f * p12, (-2.f * p12) * p11, (-2.f * p12) * p22, -2.f * p11,
                                 -2.f * p22, -4.f * p11, -4.f * p22, 0.f};
      float* base = dst + kCompBase + kPsf * kStarF + k * per * kGalF;
      if (j < nb) {
        float* o = base + j * 2 * kGalF + (dev ? 1 : 0);
#pragma unroll
        for (int e = 0; e < kGalF; ++e) o[2 * e] = vals[e];
      } else {
        const int single = dev ? (ne - nb) + (j - nb) : j - nb;
        float4* o = reinterpret_cast<float4*>(base + nb * 2 * kGalF + single * kGalF);
#pragma unroll
        for (int e = 0; e < kGalF / 4; ++e)
          o[e] = make_float4(vals[4 * e], vals[4 * e + 1], vals[4 * e + 2], vals[4 * e + 3]);
      }
    }
  }
}

// Skip radii of the staged galaxy pairs, after stage_record and a warp
// barrier (derivs layout: a pair's first eight floats are its {A11, A12, A22,
// lw}): for d^2 beyond rec[kSkipBase + k kMaxProf + j] both halves of pair
// j have log2 phi <= lw - lambda_min(-A) d^2 < -128, where exp2 (which
// flushes denormals here) returns zero, so the pair would add exact zeros.
// 0.1 % on the radius and two powers of two of slack cover the rounding of
// the bound and of the exponent; an ill-conditioned or non-finite form is
// never skipped.
__device__ __forceinline__ void stage_skip(float* __restrict__ rec, int ne, int nd, int lane) {
  const int nb = ne < nd ? ne : nd;
  if (lane < kPsf * nb) {
    const int k = lane / nb, j = lane - k * nb;
    const float* c = rec + kCompBase + kPsf * kStarF + (k * (ne + nd) + 2 * j) * kGalF;
    float r = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float a = -c[h], b = -0.5f * c[2 + h], d = -c[4 + h], lw = c[6 + h];
      const float det = fmaf(a, d, -b * b);
      const float lmax = 0.5f * (a + d + sqrtf(fmaf(a - d, a - d, 4.f * b * b)));
      const bool ok = a > 0.f && d > 0.f && det > 1e-3f * a * d && lw < INFINITY;
      r = fmaxf(r, ok ? 1.001f * fmaxf(lw + 128.f, 0.f) * (lmax / det) : INFINITY);
    }
    rec[kSkipBase + k * kMaxProf + j] = r;
  }
  __syncwarp();
}

// First pair of PSF component k that a pass over pixels with smallest squared
// offset d2 (of the whole warp) has to evaluate.
__device__ __forceinline__ int first_pair(const float* __restrict__ rec, int k, int nb, float d2,
                                          int lane) {
  const float r = rec[kSkipBase + k * kMaxProf + (lane & (kMaxProf - 1))];
  const unsigned m = __ballot_sync(0xffffffffu, lane < nb && !(d2 > r));
  return m ? __ffs(m) - 1 : nb;
}

// Smallest of the warp's squared offsets (not negative, so their bits order
// as they do; NaN orders last).
__device__ __forceinline__ float warp_min_d2(float d2) {
  return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(d2)));
}

// A pixel's offset from PSF component k's mean, and its products.
struct Offset {
  float dx, dy, xx, xy, yy;
};
__device__ __forceinline__ float2 pixel_delta(const float* __restrict__ rec, int k, float px,
                                              float py) {
  const float2 m = *reinterpret_cast<const float2*>(rec + kHdr + 2 * k);
  return make_float2(px - m.x, py - m.y);
}
__device__ __forceinline__ Offset make_offset(float2 d) {
  return Offset{d.x, d.y, d.x * d.x, d.x * d.y, d.y * d.y};
}
// Work units of a launch for one warp.  Warp w starts with unit w; with a
// queue q ([0]: units handed out beyond the first per warp, [1]: warps done;
// zero between launches) a warp then takes the next free unit whenever it
// finishes one, asking for it while it works on the current one, so every
// warp stays busy until the last unit; the last warp of the launch to finish
// resets the queue.  Without one (q null) units are dealt out by grid
// stride.  Every warp of the launch must reach done().
struct WarpQueue {
  int32_t* q;
  int it, next, stride;
  __device__ __forceinline__ WarpQueue(int32_t* queue) : q(queue), next(0) {
    stride = gridDim.x * (blockDim.x >> 5);
    it = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  }
  // at the top of every unit, before any continue
  __device__ __forceinline__ void ask(int lane) {
    if (q && lane == 0) next = stride + atomicAdd(q, 1);
  }
  __device__ __forceinline__ void advance() {
    it = q ? __shfl_sync(0xffffffffu, next, 0) : it + stride;
  }
  __device__ __forceinline__ void done(int lane) {
    if (q && lane == 0) {
      __threadfence();
      if (atomicAdd(q + 1, 1) == stride - 1) {
        q[0] = 0;
        q[1] = 0;
      }
    }
  }
};

// A lane's pixels q0, q0 + step, q0 + 2 step, ... (step 32 unless given) of
// a row-major patch of width w as (column, row), without a division per
// pixel: a step is ay rows and ax columns, plus one row when the column
// passes w.
struct PixelWalk {
  int qx, qy, ax, ay;
  __device__ __forceinline__ PixelWalk(int q0, int w, int step = 32) {
    qy = q0 / w;
    qx = q0 - qy * w;
    ay = step / w;
    ax = step - ay * w;
  }
  __device__ __forceinline__ void next(int w) {
    qx += ax;
    qy += ay;
    if (qx >= w) {
      qx -= w;
      ++qy;
    }
  }
};

// Density (weight and normaliser included) of a component with coefficients q.
__device__ __forceinline__ float gauss_density(const float4 q, const Offset& o) {
  return exp2f(fmaf(q.x, o.xx, fmaf(q.y, o.xy, fmaf(q.z, o.yy, q.w))));
}

// Sums over the components of one galaxy profile (weights without rho):
// S*: derivatives in mu; T2: tau-weighted second order (-> dG);
// T3: tau-weighted third order (-> d mu dG); T4: tau^2 fourth order (-> dG dG).
// The odd orders (s1*, t3*) are accumulated with the opposite sign: the
// kernels form z = -y = (-P) (p - mu) from the staged -P, and the Hermite
// polynomials of odd order change sign with y.
struct GalSums {
  float s0, s1x, s1y, s2xx, s2xy, s2yy;
  float t2xx, t2xy, t2yy;
  float t3a, t3b, t3c, t3d;            // 111, 112, 122, 222
  float t4a, t4b, t4c, t4d, t4e;       // 1111, 1112, 1122, 1222, 2222
};

// One galaxy component of the derivs layout (its first 16 values).
__device__ __forceinline__ void gal_accumulate(const float* __restrict__ c, const Offset& o,
                                               GalSums& g) {
  const float4 q = *reinterpret_cast<const float4*>(c);
  const float4 pp = *reinterpret_cast<const float4*>(c + 4);
  const float4 hc = *reinterpret_cast<const float4*>(c + 8);
  const float4 hd = *reinterpret_cast<const float4*>(c + 12);
  const float m4P12 = hd.x, c4b = hd.y, c4d = hd.z;
  const float nP11 = pp.x, nP12 = pp.y, nP22 = pp.z, tau = pp.w, m2P12 = hc.x;
  const float z1 = fmaf(nP11, o.dx, nP12 * o.dy);       // -y1
  const float z2 = fmaf(nP12, o.dx, nP22 * o.dy);       // -y2
  const float phi = gauss_density(q, o);
  const float h11 = fmaf(z1, z1, nP11);                 // y y^T - P
  const float h12 = fmaf(z1, z2, nP12);
  const float h22 = fmaf(z2, z2, nP22);
  const float pt = phi * tau;
  const float pt2 = pt * tau;
  g.s0 += phi;
  g.s1x = fmaf(phi, z1, g.s1x);
  g.s1y = fmaf(phi, z2, g.s1y);
  g.s2xx = fmaf(phi, h11, g.s2xx);
  g.s2xy = fmaf(phi, h12, g.s2xy);
  g.s2yy = fmaf(phi, h22, g.s2yy);
  g.t2xx = fmaf(pt, h11, g.t2xx);
  g.t2xy = fmaf(pt, h12, g.t2xy);
  g.t2yy = fmaf(pt, h22, g.t2yy);
  // third order: y_a y_b y_c - (P_ab y_c + P_ac y_b + P_bc y_a)
  const float a1 = fmaf(2.f, nP11, h11), a2 = fmaf(2.f, nP22, h22);
  const float pz1 = pt * z1, pz2 = pt * z2;
  g.t3a = fmaf(pz1, a1, g.t3a);
  g.t3b = fmaf(pz2, h11, fmaf(m2P12, pz1, g.t3b));
  g.t3c = fmaf(pz1, h22, fmaf(m2P12, pz2, g.t3c));
  g.t3d = fmaf(pz2, a2, g.t3d);
  // fourth order, written with h = y y^T - P (y1^2 = h11 + P11, y2^2 =
  // h22 + P22: the -2 P12 P terms are staged)
  g.t4a = fmaf(pt2, fmaf(h11, fmaf(4.f, nP11, h11), hc.y), g.t4a);
  g.t4b = fmaf(pt2, fmaf(h12, a1, fmaf(m2P12, h11, c4b)), g.t4b);
  g.t4c = fmaf(pt2, fmaf(h11, h22, fmaf(h12, m4P12, hc.w)), g.t4c);
  g.t4d = fmaf(pt2, fmaf(h12, a2, fmaf(m2P12, h22, c4d)), g.t4d);
  g.t4e = fmaf(pt2, fmaf(h22, fmaf(4.f, nP22, h22), hc.z), g.t4e);
}

// ---- packed pairs (exponential j, de Vaucouleurs j) ------------------------
// ffma2 / fmul2 / fadd2 round each half exactly as fmaf / * / + do, so the
// packed sums equal, bit for bit, the ones the scalar code forms.
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }

// A pixel's offset products, duplicated in both halves.
struct Offset2 {
  float2 dx, dy, xx, xy, yy;
};
__device__ __forceinline__ Offset2 dup_offset(const Offset& o) {
  return Offset2{f2(o.dx), f2(o.dy), f2(o.xx), f2(o.xy), f2(o.yy)};
}

// The sums of GalSums for both profiles: .x exponential, .y de Vaucouleurs.
struct GalSums2 {
  float2 s0, s1x, s1y, s2xx, s2xy, s2yy;
  float2 t2xx, t2xy, t2yy;
  float2 t3a, t3b, t3c, t3d;
  float2 t4a, t4b, t4c, t4d, t4e;
};

// gal_accumulate on a staged pair (40 floats, exponential in the even slots).
// Accumulations sharing phi, pt or pt2 stand together: 4.49 ms against 4.64
// in the order of the formulas (derivatives of 1,000 blended sources).
__device__ __forceinline__ void gal_accumulate2(const float* __restrict__ c, const Offset2& o,
                                                GalSums2& g) {
  const float4 qa = *reinterpret_cast<const float4*>(c);
  const float4 qb = *reinterpret_cast<const float4*>(c + 4);
  const float4 pa = *reinterpret_cast<const float4*>(c + 8);
  const float4 pb = *reinterpret_cast<const float4*>(c + 12);
  const float4 ha = *reinterpret_cast<const float4*>(c + 16);
  const float4 hb = *reinterpret_cast<const float4*>(c + 20);
  const float4 hq = *reinterpret_cast<const float4*>(c + 24);
  const float4 hr = *reinterpret_cast<const float4*>(c + 28);
  const float4 hs4 = *reinterpret_cast<const float4*>(c + 32);
  const float2 n4P22 = *reinterpret_cast<const float2*>(c + 36);
  const float2 c4d = make_float2(hr.x, hr.y), n2P11 = make_float2(hr.z, hr.w);
  const float2 n2P22 = make_float2(hs4.x, hs4.y), n4P11 = make_float2(hs4.z, hs4.w);
  const float2 m4P12 = make_float2(hq.x, hq.y), c4b = make_float2(hq.z, hq.w);
  const float2 A11 = make_float2(qa.x, qa.y), A12 = make_float2(qa.z, qa.w);
  const float2 A22 = make_float2(qb.x, qb.y), lw = make_float2(qb.z, qb.w);
  const float2 nP11 = make_float2(pa.x, pa.y), nP12 = make_float2(pa.z, pa.w);
  const float2 nP22 = make_float2(pb.x, pb.y), tau = make_float2(pb.z, pb.w);
  const float2 m2P12 = make_float2(ha.x, ha.y), c4a = make_float2(ha.z, ha.w);
  const float2 c4e = make_float2(hb.x, hb.y), c4c = make_float2(hb.z, hb.w);
  const float2 z1 = fma2(nP11, o.dx, mul2(nP12, o.dy));
  const float2 z2 = fma2(nP12, o.dx, mul2(nP22, o.dy));
  const float2 arg = fma2(A11, o.xx, fma2(A12, o.xy, fma2(A22, o.yy, lw)));
  const float2 phi = make_float2(exp2f(arg.x), exp2f(arg.y));
  const float2 h11 = fma2(z1, z1, nP11);
  const float2 h12 = fma2(z1, z2, nP12);
  const float2 h22 = fma2(z2, z2, nP22);
  const float2 pt = mul2(tau, phi);
  g.s0 = add2(phi, g.s0);
  g.s1x = fma2(phi, z1, g.s1x);
  g.s1y = fma2(phi, z2, g.s1y);
  g.s2xx = fma2(phi, h11, g.s2xx);
  g.s2xy = fma2(phi, h12, g.s2xy);
  g.s2yy = fma2(phi, h22, g.s2yy);
  const float2 pt2 = mul2(tau, pt);
  g.t2xx = fma2(pt, h11, g.t2xx);
  g.t2xy = fma2(pt, h12, g.t2xy);
  g.t2yy = fma2(pt, h22, g.t2yy);
  const float2 pz1 = mul2(pt, z1), pz2 = mul2(pt, z2);
  const float2 a1 = add2(h11, n2P11), a2 = add2(h22, n2P22);
  g.t3b = fma2(m2P12, pz1, g.t3b);
  g.t3c = fma2(m2P12, pz2, g.t3c);
  const float2 ub = fma2(m2P12, h11, c4b);
  const float2 ud = fma2(m2P12, h22, c4d);
  g.t3b = fma2(pz2, h11, g.t3b);
  g.t3d = fma2(pz2, a2, g.t3d);
  g.t3a = fma2(pz1, a1, g.t3a);
  g.t3c = fma2(pz1, h22, g.t3c);
  const float2 va = fma2(h11, add2(h11, n4P11), c4a);
  const float2 uc = fma2(h12, m4P12, c4c);
  const float2 vc = fma2(h11, h22, uc);
  const float2 ve = fma2(h22, add2(h22, n4P22), c4e);
  const float2 vb = fma2(h12, a1, ub);
  const float2 vd = fma2(h12, a2, ud);
  g.t4a = fma2(pt2, va, g.t4a);
  g.t4b = fma2(pt2, vb, g.t4b);
  g.t4c = fma2(pt2, vc, g.t4c);
  g.t4d = fma2(pt2, vd, g.t4d);
  g.t4e = fma2(pt2, ve, g.t4e);
}

// A component without a partner: gal_accumulate into half L of g.
template <int L>
__device__ __forceinline__ void gal_single(const float* __restrict__ c, const Offset& o,
                                           GalSums2& g) {
  GalSums h;
#define GET(f) h.f = L ? g.f.y : g.f.x;
#define PUT(f) (L ? g.f.y : g.f.x) = h.f;
#define ALL(M) M(s0) M(s1x) M(s1y) M(s2xx) M(s2xy) M(s2yy) M(t2xx) M(t2xy) M(t2yy) \
               M(t3a) M(t3b) M(t3c) M(t3d) M(t4a) M(t4b) M(t4c) M(t4d) M(t4e)
  ALL(GET)
  gal_accumulate(c, o, h);
  ALL(PUT)
#undef ALL
#undef PUT
#undef GET
}

// Galaxy (rho-mixed) and star profile densities of one pair at two pixels a
// and b (value layout), reading each staged component once: the galaxy pairs
// in packed two-wide instructions, the exponential and de Vaucouleurs sums in
// the two halves (each half adds its components in the order of the
// derivative kernel's sums).  (Leaving out vanished pairs, as the derivative
// kernel does, costs more than it saves here: 1.64 ms against 1.62 for a
// value pass of 2,000 blended sources, 1.40 against 1.28 for renders and
// backgrounds of 500.)
__device__ __forceinline__ void profiles_value2(const float* __restrict__ rec, int ne, int nd,
                                                float pxa, float pya, float pxb, float pyb,
                                                float& F0a, float& F1a, float& F0b, float& F1b) {
  const float4* q4 = reinterpret_cast<const float4*>(rec + kCompBase);
  float fsa = 0.f, fsb = 0.f;
  float2 fa = make_float2(0.f, 0.f), fb = make_float2(0.f, 0.f);
  const int per = ne + nd;
  const int nb = ne < nd ? ne : nd;
#pragma unroll
  for (int k = 0; k < kPsf; ++k) {
    const Offset oa = make_offset(pixel_delta(rec, k, pxa, pya));
    const Offset ob = make_offset(pixel_delta(rec, k, pxb, pyb));
    const float4 qs = q4[k];
    fsa += gauss_density(qs, oa);
    fsb += gauss_density(qs, ob);
    const Offset2 a2 = dup_offset(oa), b2 = dup_offset(ob);
    const float4* g = q4 + kPsf + k * per;
#pragma unroll 4
    for (int j = 0; j < nb; ++j) {
      const float4 a = g[2 * j], b = g[2 * j + 1];
      const float2 A11 = make_float2(a.x, a.y), A12 = make_float2(a.z, a.w);
      const float2 A22 = make_float2(b.x, b.y), lw = make_float2(b.z, b.w);
      const float2 ga = fma2(A11, a2.xx, fma2(A12, a2.xy, fma2(A22, a2.yy, lw)));
      const float2 gb = fma2(A11, b2.xx, fma2(A12, b2.xy, fma2(A22, b2.yy, lw)));
      fa = add2(fa, make_float2(exp2f(ga.x), exp2f(ga.y)));
      fb = add2(fb, make_float2(exp2f(gb.x), exp2f(gb.y)));
    }
    const float4* single = g + 2 * nb;
    for (int j = nb; j < ne; ++j, ++single) {
      fa.x += gauss_density(*single, oa);
      fb.x += gauss_density(*single, ob);
    }
    for (int j = nb; j < nd; ++j, ++single) {
      fa.y += gauss_density(*single, oa);
      fb.y += gauss_density(*single, ob);
    }
  }
  const float rho = rec[H_RHO], rho1 = rec[H_RHO1];
  F0a = fmaf(rho, fa.x, rho1 * fa.y);
  F1a = fsa;
  F0b = fmaf(rho, fb.x, rho1 * fb.y);
  F1b = fsb;
}

// The source's own E_q[l f] and V_q[l f] at a pixel.  V uses the
// cancellation-free form sum_i q_i ev_i (k_i F_i)^2 + q0 q1 (k0 F0 - k1 F1)^2.
__device__ __forceinline__ void own_moments(const float* __restrict__ rec, float F0, float F1,
                                            float& Es, float& Vs) {
  const float k0F = rec[H_K0] * F0, k1F = rec[H_K1] * F1;
  Es = fmaf(rec[H_CE0], F0, rec[H_CE1] * F1);
  const float d = k0F - k1F;
  Vs = fmaf(rec[H_Q0] * rec[H_EV0] * k0F, k0F,
            fmaf(rec[H_Q1] * rec[H_EV1] * k1F, k1F, rec[H_Q0] * rec[H_Q1] * d * d));
}

// The 52 Hessian sums of a lane live in its warp's shared memory: row a
// (the sum hidx = kGradAcc + a) of a padded [kHessAcc][33] array, this lane's
// column.  The 33-float rows keep both the per-pixel updates (one row, all
// lanes) and the transposed reduction (one row per lane) free of bank
// conflicts, and the registers this frees keep more warps resident.
constexpr int kHessAcc = kAcc - kGradAcc;   // 52
constexpr int kHessRow = 33;
constexpr int kAccTileF = kAcc * kHessRow;  // all 64 sums at the reduction

struct HessAcc {
  float* __restrict__ col;   // this lane's column of the warp's array
  __device__ __forceinline__ float* at(int idx) const { return col + (idx - kGradAcc) * kHessRow; }
  // sum += v
  __device__ __forceinline__ void add(int idx, float v) const { *at(idx) += v; }
  // sum = fma(a, b, sum)
  __device__ __forceinline__ void fma(int idx, float a, float b) const {
    float* p = at(idx);
    *p = fmaf(a, b, *p);
  }
  // sum = fma(a, b, fma(c, d, sum))
  __device__ __forceinline__ void fma2(int idx, float a, float b, float c, float d) const {
    float* p = at(idx);
    *p = fmaf(a, b, fmaf(c, d, *p));
  }
};

// The star sums of a pixel: value, d mu, d mu d mu.
struct StarSums {
  float F1, sx, sy, sxx, sxy, syy;
};

// The value and gradient sums of a lane (sums 0..11): in registers, or in the
// rows below the Hessian's of a tile in shared memory.
struct GradRegs {
  float* __restrict__ a;
  __device__ __forceinline__ void add(int i, float v) const { a[i] += v; }
  __device__ __forceinline__ void fma(int i, float x, float y) const { a[i] = fmaf(x, y, a[i]); }
  __device__ __forceinline__ void fma2(int i, float x, float y, float z, float w) const {
    a[i] = fmaf(x, y, fmaf(z, w, a[i]));
  }
};
struct GradTile {
  float* __restrict__ col;
  __device__ __forceinline__ float* at(int i) const { return col + (kHessAcc + i) * kHessRow; }
  __device__ __forceinline__ void add(int i, float v) const { *at(i) += v; }
  __device__ __forceinline__ void fma(int i, float x, float y) const { *at(i) = fmaf(x, y, *at(i)); }
  __device__ __forceinline__ void fma2(int i, float x, float y, float z, float w) const {
    *at(i) = fmaf(x, y, fmaf(z, w, *at(i)));
  }
};

// A pixel's star and galaxy sums; with kSkip for a whole warp of pixels at
// once, leaving out the pairs that are zero at all of them.
template <bool kSkip>
__device__ __forceinline__ void pixel_sums(const float* __restrict__ rec, int ne, int nd,
                                           float px, float py, int lane, StarSums& st,
                                           GalSums2& g2) {
  st = {};
#pragma unroll
  for (int k = 0; k < kPsf; ++k) {
    const Offset o = make_offset(pixel_delta(rec, k, px, py));
    const float* c = rec + kCompBase + k * kStarF;
    const float4 q = *reinterpret_cast<const float4*>(c);
    const float4 pp = *reinterpret_cast<const float4*>(c + 4);
    const float y1 = fmaf(pp.x, o.dx, pp.y * o.dy);
    const float y2 = fmaf(pp.y, o.dx, pp.z * o.dy);
    const float phi = gauss_density(q, o);
    st.F1 += phi;
    st.sx = fmaf(phi, y1, st.sx);
    st.sy = fmaf(phi, y2, st.sy);
    st.sxx = fmaf(phi, fmaf(y1, y1, -pp.x), st.sxx);
    st.sxy = fmaf(phi, fmaf(y1, y2, -pp.y), st.sxy);
    st.syy = fmaf(phi, fmaf(y2, y2, -pp.z), st.syy);
  }
  // galaxy: exponential and de Vaucouleurs sums, evaluated in pairs
  g2 = {};
  const int per = ne + nd;
  const int nb = ne < nd ? ne : nd;
  // kept rolled: three copies of this loop cost more in instruction fetch
  // than recomputing the offsets
#pragma unroll 1
  for (int k = 0; k < kPsf; ++k) {
    const float* base = rec + kCompBase + kPsf * kStarF + k * per * kGalF;
    const Offset o = make_offset(pixel_delta(rec, k, px, py));
    const Offset2 o2 = dup_offset(o);
    int j = kSkip ? first_pair(rec, k, nb, warp_min_d2(o.xx + o.yy), lane) : 0;
    if (nb == kMaxProf && j < 2) {
      // the usual eight pairs, unrolled: independent pairs interleave (the
      // loop over PSF components stays rolled: unrolling both measured
      // slower, from instruction fetch)
#pragma unroll
      for (int jj = 0; jj < kMaxProf; ++jj) gal_accumulate2(base + jj * 2 * kGalF, o2, g2);
    } else {
#pragma unroll 2
      for (; j < nb; ++j) gal_accumulate2(base + j * 2 * kGalF, o2, g2);
    }
    const float* single = base + nb * 2 * kGalF;
    for (int j = nb; j < ne; ++j, single += kGalF) gal_single<0>(single, o, g2);
    for (int j = nb; j < nd; ++j, single += kGalF) gal_single<1>(single, o, g2);
  }
}

// One pixel with its sums: accumulates value, gradient and Hessian.  With
// kTurn every term is formed before turn() is called and added after it, if
// it returns true.
template <bool kTurn, class G, class T>
__device__ __forceinline__ void pixel_derivs(const float* __restrict__ rec, const StarSums& st,
                                             const GalSums2& g2, float x, float2 bg, const G& acc,
                                             const HessAcc& hs, T&& turn) {
  const float F1 = st.F1, sx = st.sx, sy = st.sy, sxx = st.sxx, sxy = st.sxy, syy = st.syy;
  GalSums ge, gd;
#define SPLIT(f) ge.f = g2.f.x; gd.f = g2.f.y;
#define FLIP(f) ge.f = -g2.f.x; gd.f = -g2.f.y;        // odd orders: summed with -y
  SPLIT(s0) FLIP(s1x) FLIP(s1y) SPLIT(s2xx) SPLIT(s2xy) SPLIT(s2yy) SPLIT(t2xx) SPLIT(t2xy)
  SPLIT(t2yy) FLIP(t3a) FLIP(t3b) FLIP(t3c) FLIP(t3d) SPLIT(t4a) SPLIT(t4b) SPLIT(t4c)
  SPLIT(t4d) SPLIT(t4e)
#undef FLIP
#undef SPLIT
  const float rho = rec[H_RHO], rho1 = rec[H_RHO1];
#define MIX(f) fmaf(rho, ge.f, rho1 * gd.f)
  // galaxy density and its derivatives over (mu_x, mu_y, g11, g12, g22, rho)
  const float F0 = MIX(s0);
  float d0[6], h0[6][6];
  d0[0] = MIX(s1x);
  d0[1] = MIX(s1y);
  d0[2] = 0.5f * MIX(t2xx);
  d0[3] = MIX(t2xy);
  d0[4] = 0.5f * MIX(t2yy);
  d0[5] = ge.s0 - gd.s0;
  h0[0][0] = MIX(s2xx);
  h0[0][1] = MIX(s2xy);
  h0[1][1] = MIX(s2yy);
  h0[0][2] = 0.5f * MIX(t3a);
  h0[1][2] = 0.5f * MIX(t3b);
  h0[0][3] = MIX(t3b);
  h0[1][3] = MIX(t3c);
  h0[0][4] = 0.5f * MIX(t3c);
  h0[1][4] = 0.5f * MIX(t3d);
  h0[2][2] = 0.25f * MIX(t4a);
  h0[2][3] = 0.5f * MIX(t4b);
  h0[2][4] = 0.25f * MIX(t4c);
  h0[3][3] = MIX(t4c);
  h0[3][4] = 0.5f * MIX(t4d);
  h0[4][4] = 0.25f * MIX(t4e);
  h0[0][5] = ge.s1x - gd.s1x;
  h0[1][5] = ge.s1y - gd.s1y;
  h0[2][5] = 0.5f * (ge.t2xx - gd.t2xx);
  h0[3][5] = ge.t2xy - gd.t2xy;
  h0[4][5] = 0.5f * (ge.t2yy - gd.t2yy);
  h0[5][5] = 0.f;
#undef MIX

  // ---- moments and the pixel term
  const float cE0 = rec[H_CE0], cE1 = rec[H_CE1], cM0 = rec[H_CM0], cM1 = rec[H_CM1];
  float Es, Vs;
  own_moments(rec, F0, F1, Es, Vs);
  const float bgE = bg.x, bgV = bg.y;
  const float E = bgE + Es, V = bgV + Vs;
  const float r = __frcp_rn(E);
  const float rb = __frcp_rn(bgE);
  const float xr = x * r;
  const float xr2 = xr * r;        // x / E^2
  const float xr3 = xr2 * r;       // x / E^3
  const float TE = fmaf(x - E, r, xr3 * V);
  const float TV = -0.5f * xr2;
  const float TEE = fmaf(-3.f * xr3 * r, V, -xr2);
  const float TEV = xr3;
  const float tE = fmaf(-2.f * Es, TV, TE);
  const float tM = TV;
  const float tEE = fmaf(-4.f * Es, TEV, fmaf(-2.f, TV, TEE));
  const float tEM = TEV;

  const float v_rel = fmaf(x, log1pf(Es * rb) - 0.5f * V * r * r + 0.5f * bgV * rb * rb, -Es);
  const float v_base = fmaf(x, __logf(bgE) - 0.5f * bgV * rb * rb, -bgE);

  // gradient vectors of E_s (a) and M_s (b) over the six geometric coordinates
  float aG[6], bG[6];
  const float m0 = 2.f * cM0 * F0, m1 = 2.f * cM1 * F1;
  aG[0] = fmaf(cE0, d0[0], cE1 * sx);
  aG[1] = fmaf(cE0, d0[1], cE1 * sy);
  bG[0] = fmaf(m0, d0[0], m1 * sx);
  bG[1] = fmaf(m0, d0[1], m1 * sy);
#pragma unroll
  for (int g = 2; g < 6; ++g) {
    aG[g] = cE0 * d0[g];
    bG[g] = m0 * d0[g];
  }
  const float F0s = F0 * F0, F1s = F1 * F1;
  // Hessian: tEE a a^T + tEM (a b^T + b a^T) + tE d2E_s + tM d2M_s
  float u[6], cg[6];
#pragma unroll
  for (int g = 0; g < 6; ++g) {
    cg[g] = tEM * bG[g];
    u[g] = fmaf(tEE, aG[g], cg[g]);
  }
  const float tm2F0 = 2.f * tM * F0, tm2F1 = 2.f * tM * F1;
  const float eF0 = tEM * F0s, eF1 = tEM * F1s;
  const float D0 = fmaf(tE, cE0, tM * m0);   // dl/dF0 (direct part)
  const float D1 = fmaf(tE, cE1, tM * m1);
  const float q0 = 2.f * tM * cM0, q1 = 2.f * tM * cM1;
  const float h1[2][2] = {{sxx, sxy}, {sxy, syy}};
  const float d1[2] = {sx, sy};
  auto geo = [&](int g, int h) {
    float v = fmaf(aG[g], u[h], cg[g] * aG[h]);
    v = fmaf(D0, h0[g][h], v);
    v = fmaf(q0 * d0[g], d0[h], v);
    if (g < 2 && h < 2) {
      v = fmaf(D1, h1[g][h], v);
      v = fmaf(q1 * d1[g], d1[h], v);
    }
    return v;
  };
  float vv[kTurn ? 36 : 1];
  if (kTurn) {
#pragma unroll
    for (int g = 0; g < 6; ++g)
#pragma unroll
      for (int h = g; h < 6; ++h) vv[kTurn ? 6 * g + h : 0] = geo(g, h);
  }
  if (!turn()) return;
  acc.add(0, v_rel);
  acc.add(1, v_base);
  // gradient over w
  acc.fma(2, tE, F0);
  acc.fma(3, tE, F1);
  acc.fma(4, tM, F0s);
  acc.fma(5, tM, F1s);
#pragma unroll
  for (int g = 0; g < 6; ++g) acc.fma2(6 + g, tE, aG[g], tM, bG[g]);
  hs.fma(hidx(0, 0), tEE, F0s);
  hs.fma(hidx(0, 1), tEE, F0 * F1);
  hs.fma(hidx(1, 1), tEE, F1s);
  hs.fma(hidx(0, 2), tEM * F0, F0s);
  hs.fma(hidx(0, 3), tEM * F0, F1s);
  hs.fma(hidx(1, 2), tEM * F1, F0s);
  hs.fma(hidx(1, 3), tEM * F1, F1s);
#pragma unroll
  for (int g = 0; g < 6; ++g) {
    hs.fma2(hidx(0, 4 + g), F0, u[g], tE, d0[g]);
    hs.fma2(hidx(2, 4 + g), eF0, aG[g], tm2F0, d0[g]);
  }
  hs.fma2(hidx(1, 4), F1, u[0], tE, sx);
  hs.fma2(hidx(1, 5), F1, u[1], tE, sy);
  hs.fma2(hidx(3, 4), eF1, aG[0], tm2F1, sx);
  hs.fma2(hidx(3, 5), eF1, aG[1], tm2F1, sy);
#pragma unroll
  for (int g = 2; g < 6; ++g) {
    hs.fma(hidx(1, 4 + g), F1, u[g]);
    hs.fma(hidx(3, 4 + g), eF1, aG[g]);
  }
#pragma unroll
  for (int g = 0; g < 6; ++g)
#pragma unroll
    for (int h = g; h < 6; ++h) hs.add(hidx(4 + g, 4 + h), kTurn ? vv[kTurn ? 6 * g + h : 0] : geo(g, h));
}

// Gradient-only sums of one galaxy profile: value, d mu, and the
// tau-weighted second order for dG (the heat equation again).
struct GalSums1 {
  float s0, s1x, s1y, t2xx, t2xy, t2yy;
};

__device__ __forceinline__ void gal_accumulate1(const float* __restrict__ c, const Offset& o,
                                                GalSums1& g) {
  const float4 q = *reinterpret_cast<const float4*>(c);
  const float4 pp = *reinterpret_cast<const float4*>(c + 4);
  const float nP11 = pp.x, nP12 = pp.y, nP22 = pp.z;
  const float z1 = fmaf(nP11, o.dx, nP12 * o.dy);       // -y1
  const float z2 = fmaf(nP12, o.dx, nP22 * o.dy);
  const float phi = gauss_density(q, o);
  const float pt = phi * pp.w;
  g.s0 += phi;
  g.s1x = fmaf(phi, z1, g.s1x);
  g.s1y = fmaf(phi, z2, g.s1y);
  g.t2xx = fmaf(pt, fmaf(z1, z1, nP11), g.t2xx);
  g.t2xy = fmaf(pt, fmaf(z1, z2, nP12), g.t2xy);
  g.t2yy = fmaf(pt, fmaf(z2, z2, nP22), g.t2yy);
}

struct GalSums1x2 {
  float2 s0, s1x, s1y, t2xx, t2xy, t2yy;
};

// gal_accumulate1 on a staged pair (exponential in the even slots).
__device__ __forceinline__ void gal_accumulate1x2(const float* __restrict__ c, const Offset2& o,
                                                  GalSums1x2& g) {
  const float4 qa = *reinterpret_cast<const float4*>(c);
  const float4 qb = *reinterpret_cast<const float4*>(c + 4);
  const float4 pa = *reinterpret_cast<const float4*>(c + 8);
  const float4 pb = *reinterpret_cast<const float4*>(c + 12);
  const float2 A11 = make_float2(qa.x, qa.y), A12 = make_float2(qa.z, qa.w);
  const float2 A22 = make_float2(qb.x, qb.y), lw = make_float2(qb.z, qb.w);
  const float2 nP11 = make_float2(pa.x, pa.y), nP12 = make_float2(pa.z, pa.w);
  const float2 nP22 = make_float2(pb.x, pb.y), tau = make_float2(pb.z, pb.w);
  const float2 z1 = fma2(nP11, o.dx, mul2(nP12, o.dy));
  const float2 z2 = fma2(nP12, o.dx, mul2(nP22, o.dy));
  const float2 arg = fma2(A11, o.xx, fma2(A12, o.xy, fma2(A22, o.yy, lw)));
  const float2 phi = make_float2(exp2f(arg.x), exp2f(arg.y));
  const float2 pt = mul2(phi, tau);
  g.s0 = add2(g.s0, phi);
  g.s1x = fma2(phi, z1, g.s1x);
  g.s1y = fma2(phi, z2, g.s1y);
  g.t2xx = fma2(pt, fma2(z1, z1, nP11), g.t2xx);
  g.t2xy = fma2(pt, fma2(z1, z2, nP12), g.t2xy);
  g.t2yy = fma2(pt, fma2(z2, z2, nP22), g.t2yy);
}

template <int L>
__device__ __forceinline__ void gal_single1(const float* __restrict__ c, const Offset& o,
                                            GalSums1x2& g) {
  GalSums1 h;
#define GET(f) h.f = L ? g.f.y : g.f.x;
#define PUT(f) (L ? g.f.y : g.f.x) = h.f;
#define ALL(M) M(s0) M(s1x) M(s1y) M(t2xx) M(t2xy) M(t2yy)
  ALL(GET)
  gal_accumulate1(c, o, h);
  ALL(PUT)
#undef ALL
#undef PUT
#undef GET
}

// One pixel, value and gradient only (the adjoint of the pixel term through
// E_s and M_s onto the per-image natural coordinates): 12 accumulators.
__device__ __forceinline__ void pixel_grad(const float* __restrict__ rec, int ne, int nd,
                                           float px, float py, float x, float2 bg,
                                           float* __restrict__ acc) {
  float F1 = 0.f, sx = 0.f, sy = 0.f;
  float2 dk[kPsf];
#pragma unroll
  for (int k = 0; k < kPsf; ++k) {
    dk[k] = pixel_delta(rec, k, px, py);
    const Offset o = make_offset(dk[k]);
    const float* c = rec + kCompBase + k * kStarF;
    const float4 q = *reinterpret_cast<const float4*>(c);
    const float4 pp = *reinterpret_cast<const float4*>(c + 4);
    const float y1 = fmaf(pp.x, o.dx, pp.y * o.dy);
    const float y2 = fmaf(pp.y, o.dx, pp.z * o.dy);
    const float phi = gauss_density(q, o);
    F1 += phi;
    sx = fmaf(phi, y1, sx);
    sy = fmaf(phi, y2, sy);
  }
  GalSums1x2 g2 = {};
  const int per = ne + nd;
  const int nb = ne < nd ? ne : nd;
#pragma unroll
  for (int k = 0; k < kPsf; ++k) {
    const float* base = rec + kCompBase + kPsf * kStarF + k * per * kGalF;
    const Offset o = make_offset(dk[k]);
    const Offset2 o2 = dup_offset(o);
    for (int j = 0; j < nb; ++j) gal_accumulate1x2(base + j * 2 * kGalF, o2, g2);
    const float* single = base + nb * 2 * kGalF;
    for (int j = nb; j < ne; ++j, single += kGalF) gal_single1<0>(single, o, g2);
    for (int j = nb; j < nd; ++j, single += kGalF) gal_single1<1>(single, o, g2);
  }
  GalSums1 ge, gd;
#define SPLIT(f) ge.f = g2.f.x; gd.f = g2.f.y;
#define FLIP(f) ge.f = -g2.f.x; gd.f = -g2.f.y;        // first order: summed with -y
  SPLIT(s0) FLIP(s1x) FLIP(s1y) SPLIT(t2xx) SPLIT(t2xy) SPLIT(t2yy)
#undef FLIP
#undef SPLIT
  const float rho = rec[H_RHO], rho1 = rec[H_RHO1];
#define MIX(f) fmaf(rho, ge.f, rho1 * gd.f)
  const float F0 = MIX(s0);
  float d0[6];
  d0[0] = MIX(s1x);
  d0[1] = MIX(s1y);
  d0[2] = 0.5f * MIX(t2xx);
  d0[3] = MIX(t2xy);
  d0[4] = 0.5f * MIX(t2yy);
  d0[5] = ge.s0 - gd.s0;
#undef MIX
  const float cE0 = rec[H_CE0], cE1 = rec[H_CE1], cM0 = rec[H_CM0], cM1 = rec[H_CM1];
  float Es, Vs;
  own_moments(rec, F0, F1, Es, Vs);
  const float bgE = bg.x, bgV = bg.y;
  const float E = bgE + Es, V = bgV + Vs;
  const float r = __frcp_rn(E);
  const float rb = __frcp_rn(bgE);
  const float xr2 = x * r * r;
  const float TE = fmaf(x - E, r, xr2 * r * V);
  const float TV = -0.5f * xr2;
  const float tE = fmaf(-2.f * Es, TV, TE);
  const float tM = TV;
  acc[0] += fmaf(x, log1pf(Es * rb) - 0.5f * V * r * r + 0.5f * bgV * rb * rb, -Es);
  acc[1] += fmaf(x, __logf(bgE) - 0.5f * bgV * rb * rb, -bgE);
  const float m0 = 2.f * cM0 * F0, m1 = 2.f * cM1 * F1;
  acc[2] = fmaf(tE, F0, acc[2]);
  acc[3] = fmaf(tE, F1, acc[3]);
  acc[4] = fmaf(tM, F0 * F0, acc[4]);
  acc[5] = fmaf(tM, F1 * F1, acc[5]);
  const float a0 = fmaf(cE0, d0[0], cE1 * sx), a1 = fmaf(cE0, d0[1], cE1 * sy);
  const float b0 = fmaf(m0, d0[0], m1 * sx), b1 = fmaf(m0, d0[1], m1 * sy);
  acc[6] = fmaf(tE, a0, fmaf(tM, b0, acc[6]));
  acc[7] = fmaf(tE, a1, fmaf(tM, b1, acc[7]));
  const float cg = fmaf(tE, cE0, tM * m0);
#pragma unroll
  for (int g = 2; g < 6; ++g) acc[6 + g] = fmaf(cg, d0[g], acc[6 + g]);
}

// Warp-shared memory of the derivative kernel: the staged record, then the
// [kAcc][kHessRow] sums (rows 0..51 the Hessian sums, rows 52..63 the value
// and gradient sums, written there for the final reduction).
constexpr int kDerivWarpF = kDerivRecF + kAccTileF;


// Sum o of an item over the lanes, along its row of the tile, in lane order,
// four chains.
__device__ __forceinline__ float row_sum(const float* __restrict__ tile, int o) {
  const float* r = tile + (o < kGradAcc ? kHessAcc + o : o - kGradAcc) * kHessRow;
  float c0 = 0.f, c1 = 0.f, c2 = 0.f, c3 = 0.f;
#pragma unroll
  for (int k = 0; k < 32; k += 4) {
    c0 += r[k];
    c1 += r[k + 1];
    c2 += r[k + 2];
    c3 += r[k + 3];
  }
  return (c0 + c1) + (c2 + c3);
}

// Adds the 64 sums of an item over the warp's lanes and writes them.  The
// two value sums take the shuffle tree every pixel kernel uses for its value
// sums, so that the value of an evaluation is the same in every pass (the
// trust-region ratio compares values of the derivative and value passes);
// for the other 62, lane l adds up rows (sums l and l + 32) along the
// 33-float rows, in lane order, four chains per row.
__device__ __forceinline__ void reduce_tile(float* __restrict__ tile, float* __restrict__ acc,
                                            float* __restrict__ out, int lane) {
#pragma unroll
  for (int a = 2; a < kGradAcc; ++a) tile[(kHessAcc + a) * kHessRow + lane] = acc[a];
  const float v0 = warp_sum(acc[0]), v1 = warp_sum(acc[1]);
  if (lane == 0) {
    out[0] = v0;
    out[1] = v1;
  }
  __syncwarp();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int o = lane + 32 * h;
    if (o >= 2) out[o] = row_sum(tile, o);
  }
}

// Four blocks of four warps per SM: with the Hessian sums in shared memory
// the kernel fits 128 registers a thread, and 16 warps keep the FP32 pipe
// fed.  (Forming the background here instead of in background_kernel was
// measured slower: the cached-moment loads inside the pixel loop stall 16
// warps more than a separate kernel's many warps.)
template <bool kQueue, bool kSkip>
__global__ void __launch_bounds__(128, 4) derivs_kernel(PlanView v, int ne, int nd) {
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  float* rec = smem + wib * kDerivWarpF;
  float* tile = rec + kDerivRecF;
  const HessAcc hs{tile + lane};
  WarpQueue wq(kQueue ? v.work_ctr : nullptr);
  for (; wq.it < v.n_items; wq.advance()) {
    wq.ask(lane);
    const int it = wq.it;
    const Item item = v.items[it];
    const PairInfo pi = v.pairs[item.pair];
    if (!v.active[pi.slot]) continue;
    __syncwarp();
    stage_record<true>(rec, v.records + (size_t)item.pair * kRecF,
                       kPsf * (1 + ne + nd), lane, ne);
#pragma unroll
    for (int a = 0; a < kHessAcc; ++a) tile[a * kHessRow + lane] = 0.f;
    __syncwarp();
    if (kSkip) stage_skip(rec, ne, nd, lane);
    float acc[kGradAcc];
#pragma unroll
    for (int a = 0; a < kGradAcc; ++a) acc[a] = 0.f;
    const int end = item.start + item.count;
    PixelWalk pw(item.start + lane, pi.w);
    // with kSkip the whole warp takes every pass, and lanes past the end
    // repeat lane 0's pixel
    for (int q = item.start + lane; (kSkip ? q - lane : q) < end; q += 32, pw.next(pi.w)) {
      int qy = pw.qy, qx = pw.qx;
      if (kSkip && q - lane + 32 > end) {
        const int y0 = __shfl_sync(0xffffffffu, qy, 0), x0 = __shfl_sync(0xffffffffu, qx, 0);
        if (q >= end) qy = y0, qx = x0;
      }
      const float x = __ldg(v.pixels + pi.pix_base + (int64_t)qy * pi.stride + qx);
      const float2 bg = v.bg[pi.bg_base + (!kSkip || q < end ? q : q - lane)];
      StarSums st;
      GalSums2 g2;
      pixel_sums<kSkip>(rec, ne, nd, (float)qx, (float)qy, lane, st, g2);
      if (!kSkip || q < end) pixel_derivs<false>(rec, st, g2, x, bg, GradRegs{acc}, hs, [] { return true; });
    }
    __syncwarp();
    reduce_tile(tile, acc, v.partials + (size_t)it * kAcc, lane);
  }
  wq.done(lane);
}

// The derivative kernel for launches too small to fill the GPU: a block of
// eight warps per item, a warp per pass of 32 pixels.  Where the kernel
// above takes an item's eight passes one after another in one warp (one
// source of 41 x 41 pixels per band: 35 warps on the whole GPU, each bound by
// its own latencies), here the warps form their pixels' sums and terms side
// by side and add them to the block's tile in pass order, handing the tile
// on through named barriers, so that every sum adds up as it does there.
// Two blocks per SM (128 registers).
constexpr int kCoopWarps = 8;
constexpr int kCoopThreads = 32 * kCoopWarps;

__global__ void __launch_bounds__(kCoopThreads, 2) derivs_coop_kernel(PlanView v, int ne, int nd) {
  __shared__ alignas(16) float rec[kDerivRecF];
  __shared__ float tile[kAccTileF];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int it = blockIdx.x;
  const Item item = v.items[it];
  const PairInfo pi = v.pairs[item.pair];
  if (!v.active[pi.slot]) return;
  if (wib == 0)
    stage_record<true>(rec, v.records + (size_t)item.pair * kRecF, kPsf * (1 + ne + nd), lane, ne);
  for (int e = threadIdx.x; e < kAccTileF; e += kCoopThreads) tile[e] = 0.f;
  __syncthreads();
  const HessAcc hs{tile + lane};
  const GradTile ga{tile + lane};
  const int end = item.start + item.count;
  PixelWalk pw(item.start + threadIdx.x, pi.w, kCoopThreads);
  for (int base = item.start; base < end; base += kCoopThreads, pw.next(pi.w)) {
    const int q = base + threadIdx.x;
    // warp w adds after warp w - 1 (barrier w), whole warps meeting there:
    // lanes past the end repeat the item's first pixel and add nothing.  The
    // rounds of an item longer than a block follow each other through the
    // block barrier below.
    auto turn = [&] {
      if (wib > 0) named_sync(wib, 64);
      return q < end;
    };
    if (base + 32 * wib < end) {
      const bool in = q < end;
      const int qx = in ? pw.qx : item.start % pi.w, qy = in ? pw.qy : item.start / pi.w;
      const float x = __ldg(v.pixels + pi.pix_base + (int64_t)qy * pi.stride + qx);
      const float2 bg = v.bg[pi.bg_base + (in ? q : item.start)];
      StarSums st;
      GalSums2 g2;
      pixel_sums<false>(rec, ne, nd, (float)qx, (float)qy, lane, st, g2);
      pixel_derivs<true>(rec, st, g2, x, bg, ga, hs, turn);
    } else {
      turn();
    }
    if (wib < kCoopWarps - 1) named_arrive(wib + 1, 64);
    if (base + kCoopThreads < end) __syncthreads();
  }
  __syncthreads();
  // the reduction over lanes, as in reduce_tile: a row a thread (warps 0, 1),
  // the value sums on the shuffle tree (warp 2)
  float* out = v.partials + (size_t)it * kAcc;
  const int o = threadIdx.x;
  if (o >= 2 && o < kAcc) {
    out[o] = row_sum(tile, o);
  } else if (wib == 2) {
    const float v0 = warp_sum(*ga.at(0)), v1 = warp_sum(*ga.at(1));
    if (lane == 0) {
      out[0] = v0;
      out[1] = v1;
    }
  }
}

template <bool kQueue>
__global__ void __launch_bounds__(128) grad_kernel(PlanView v, int ne, int nd) {
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  float* rec = smem + wib * kDerivRecF;
  WarpQueue wq(kQueue ? v.work_ctr : nullptr);
  for (; wq.it < v.n_items; wq.advance()) {
    wq.ask(lane);
    const int it = wq.it;
    const Item item = v.items[it];
    const PairInfo pi = v.pairs[item.pair];
    if (!v.active[pi.slot]) continue;
    __syncwarp();
    stage_record<true>(rec, v.records + (size_t)item.pair * kRecF,
                       kPsf * (1 + ne + nd), lane, ne);
    __syncwarp();
    float acc[kGradAcc];
#pragma unroll
    for (int a = 0; a < kGradAcc; ++a) acc[a] = 0.f;
    const int end = item.start + item.count;
    PixelWalk pw(item.start + lane, pi.w);
    for (int q = item.start + lane; q < end; q += 32, pw.next(pi.w)) {
      const int qy = pw.qy, qx = pw.qx;
      const float x = __ldg(v.pixels + pi.pix_base + (int64_t)qy * pi.stride + qx);
      const float2 bg = v.bg[pi.bg_base + q];
      pixel_grad(rec, ne, nd, (float)qx, (float)qy, x, bg, acc);
    }
#pragma unroll
    for (int a = 0; a < kGradAcc; ++a) acc[a] = warp_sum(acc[a]);
    float* out = v.partials + (size_t)it * kAcc;
#pragma unroll
    for (int a = 0; a < kGradAcc; ++a)
      if (a == lane) out[a] = acc[a];
  }
  wq.done(lane);
}

// Stages a record for value-only passes.
__device__ __forceinline__ void stage_value(float* rec, const PlanView& v, int pair, int lane,
                                            int ne, int nd) {
  __syncwarp();
  stage_record<false>(rec, v.records + (size_t)pair * kRecF, kPsf * (1 + ne + nd), lane, ne);
  __syncwarp();
}

// The own moments at pixels [begin, end) (row-major) of a rectangle w
// columns wide: f(pre(q, column, row), q, column, row, E, V) for each, a
// lane's pixels in ascending order; pre runs before the densities are
// formed, so that what it loads is on its way meanwhile.  A lane takes pixels q and q + 32 in one pass over the
// staged components.  The whole warp takes every pass; lanes past the end
// repeat lane 0's pixel.  dx, dy: from the rectangle to the record's frame.
template <class P, class F>
__device__ __forceinline__ void for_moments(const float* __restrict__ rec, int begin, int end, int w,
                                            int dx, int dy, int lane, int ne, int nd, P&& pre,
                                            F&& f) {
  PixelWalk pa(begin + lane, w, 64), pb(begin + lane + 32, w, 64);
  for (int q = begin + lane; q - lane < end; q += 64, pa.next(w), pb.next(w)) {
    int xa = pa.qx, ya = pa.qy, xb = pb.qx, yb = pb.qy;
    if (q - lane + 64 > end) {
      const int x0 = __shfl_sync(0xffffffffu, xa, 0), y0 = __shfl_sync(0xffffffffu, ya, 0);
      if (q >= end) xa = x0, ya = y0;
      if (q + 32 >= end) xb = x0, yb = y0;
    }
    const bool in_a = q < end, in_b = q + 32 < end;
    const auto la = pre(in_a ? q : q - lane, xa, ya), lb = pre(in_b ? q + 32 : q - lane, xb, yb);
    float F0[2], F1[2];
    profiles_value2(rec, ne, nd, (float)(xa + dx), (float)(ya + dy), (float)(xb + dx),
                    (float)(yb + dy), F0[0], F1[0], F0[1], F1[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (q + 32 * h >= end) break;
      float Es, Vs;
      own_moments(rec, F0[h], F1[h], Es, Vs);
      f(h ? lb : la, q + 32 * h, h ? xb : xa, h ? yb : ya, Es, Vs);
    }
  }
}

// The pixel term relative to the source's absence, and without the source.
__device__ __forceinline__ float2 value_term(float x, float2 bg, float Es, float Vs) {
  const float E = bg.x + Es, V = bg.y + Vs;
  const float r = __frcp_rn(E), rb = __frcp_rn(bg.x);
  return make_float2(fmaf(x, log1pf(Es * rb) - 0.5f * V * r * r + 0.5f * bg.y * rb * rb, -Es),
                     fmaf(x, __logf(bg.x) - 0.5f * bg.y * rb * rb, -bg.x));
}

// Where a value pass with keep_render keeps the own moments: 0 nowhere; 1 in
// v.trial_render; 2 in the source's other half of the render cache (where a
// Newton step's trial render waits for the accept rule).
__device__ __forceinline__ float2* render_target(const PlanView& v, const PairInfo& pi,
                                                 int keep_render) {
  if (keep_render == 1) return v.trial_render + pi.bg_base;
  if (keep_render == 2)
    return v.cache + (cache_base(v, pi.source) ? 0 : v.cache_n_pool) +
           v.patches[pi.patch].pool_offset;
  return nullptr;
}

// Value-only pass over one item: the pixel term at the record's point
// (relative and baseline sums into the item's slot of vpartials); with
// render set, the own moments are also stored there (row-major over the
// patch, item pixels only).
__device__ __forceinline__ void value_item(const PlanView& v, int it, const Item& item,
                                           const PairInfo& pi, float* rec, int lane, int ne,
                                           int nd, float2* render) {
  stage_value(rec, v, item.pair, lane, ne, nd);
  float rel = 0.f, base = 0.f;
  for_moments(rec, item.start, item.start + item.count, pi.w, 0, 0, lane, ne, nd,
                     [&](int q, int qx, int qy) {
    const float2 bg = v.bg[pi.bg_base + q];
    return make_float3(__ldg(v.pixels + pi.pix_base + (int64_t)qy * pi.stride + qx), bg.x, bg.y);
  }, [&](float3 in, int q, int, int, float Es, float Vs) {
    if (render) render[q] = make_float2(Es, Vs);
    const float2 t = value_term(in.x, make_float2(in.y, in.z), Es, Vs);
    rel += t.x;
    base += t.y;
  });
  rel = warp_sum(rel);
  base = warp_sum(base);
  if (lane == 0) {
    v.vpartials[2 * (size_t)it] = rel;
    v.vpartials[2 * (size_t)it + 1] = base;
  }
}

// Eight blocks per SM (64 registers): 3.5 % faster than seven at 72.
template <bool kQueue>
__global__ void __launch_bounds__(128, 8) value_kernel(PlanView v, int ne, int nd,
                                                    int keep_render) {
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  float* rec = smem + wib * kValRecF;
  WarpQueue wq(kQueue ? v.work_ctr : nullptr);
  for (; wq.it < v.n_items; wq.advance()) {
    wq.ask(lane);
    const int it = wq.it;
    const Item item = v.items[it];
    const PairInfo pi = v.pairs[item.pair];
    if (!v.active[pi.slot]) continue;
    value_item(v, it, item, pi, rec, lane, ne, nd, render_target(v, pi, keep_render));
  }
  wq.done(lane);
}

// The value pass of a small launch, a block of eight warps per item and a
// warp per pass of 32 pixels; each lane's terms are then added in pass order.
__global__ void __launch_bounds__(kCoopThreads) value_coop_kernel(PlanView v, int ne, int nd,
                                                                  int keep_render) {
  __shared__ alignas(16) float rec[kValRecF];
  __shared__ float2 term[kCoopThreads];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int it = blockIdx.x;
  const Item item = v.items[it];
  const PairInfo pi = v.pairs[item.pair];
  if (!v.active[pi.slot]) return;
  float2* render = render_target(v, pi, keep_render);
  if (wib == 0)
    stage_record<false>(rec, v.records + (size_t)item.pair * kRecF, kPsf * (1 + ne + nd), lane, ne);
  __syncthreads();
  const int end = item.start + item.count;
  float rel = 0.f, base = 0.f;
  PixelWalk pw(item.start + threadIdx.x, pi.w, kCoopThreads);
  for (int b = item.start; b < end; b += kCoopThreads, pw.next(pi.w)) {
    const int q = b + threadIdx.x;
    if (q < end) {
      const float x = __ldg(v.pixels + pi.pix_base + (int64_t)pw.qy * pi.stride + pw.qx);
      const float2 bg = v.bg[pi.bg_base + q];
      float F0, F1, G0, G1, Es, Vs;
      profiles_value2(rec, ne, nd, (float)pw.qx, (float)pw.qy, (float)pw.qx, (float)pw.qy, F0, F1,
                      G0, G1);
      own_moments(rec, F0, F1, Es, Vs);
      if (render) render[q] = make_float2(Es, Vs);
      term[threadIdx.x] = value_term(x, bg, Es, Vs);
    }
    __syncthreads();
    if (wib == 0) {
#pragma unroll
      for (int k = 0; k < kCoopWarps; ++k) {
        if (b + 32 * k + lane < end) {
          rel += term[32 * k + lane].x;
          base += term[32 * k + lane].y;
        }
      }
    }
    if (b + kCoopThreads < end) __syncthreads();
  }
  if (wib == 0) {
    rel = warp_sum(rel);
    base = warp_sum(base);
    if (lane == 0) {
      v.vpartials[2 * (size_t)it] = rel;
      v.vpartials[2 * (size_t)it + 1] = base;
    }
  }
}

// ---- backgrounds, kBgChunk pixels of an item at a time: sky plus each
// neighbour's E and V where the pixel lies in that neighbour's patch (support
// rule, Sec. 2.2.3), in neighbour order.
constexpr int kBgChunk = 256;
constexpr int kBgWarpF = kValRecF + 2 * kBgChunk;          // a staged record, the chunk's sums
constexpr int kBgStages = 4;
constexpr int kBgCacheF = kBgStages * 2 * kBgChunk;        // cached moments on their way in

__device__ __forceinline__ float sky_checked(const PlanView& v, const celeste_image& im, float x,
                                             float y) {
  const float s = sky_value(im, v.sky, x, y);
  if (!(s > 0.f)) set_error(v.err, CELESTE_DERR_SKY);
  return s;
}

// Without a render cache the neighbours are rendered: the lanes go over the
// pixels of each neighbour's overlap with the chunk, two a lane (not over
// the chunk, where lanes outside the overlap would idle, nor over its whole
// rows: two overlapping patches of 1,000 x 1,000 pixels 57 us, 102 that way),
// and add to sums in the warp's shared memory (rec: kBgWarpF floats).  300
// blended sources:
// 755 us, 1,008 with a pixel a lane over the whole chunk and sums in L2; the
// 1,024 sources of a field 68 -> 42 us.
__device__ __forceinline__ void background_rendered(const PlanView& v, const Item& item,
                                                    const PairInfo& pi, float* rec, int lane,
                                                    int ne, int nd) {
  const celeste_image& im = v.images[pi.image];
  float2* sum = reinterpret_cast<float2*>(rec + kValRecF);
  const int end = item.start + item.count;
  const int nn = pi.nbr_end - pi.nbr_begin;
  for (int c0 = item.start; c0 < end; c0 += kBgChunk) {
    const int c1 = min(c0 + kBgChunk, end);
    __syncwarp();
    PixelWalk pw(c0 + lane, pi.w);
    for (int q = c0 + lane; q < c1; q += 32, pw.next(pi.w))
      sum[q - c0] =
          make_float2(sky_checked(v, im, (float)(pi.x0 + pw.qx), (float)(pi.y0 + pw.qy)), 0.f);
    for (int g0 = 0; g0 < nn; g0 += 32) {
      // the overlaps of up to 32 neighbours, one in each lane
      int np = 0, nx = 0, ny = 0;
      Overlap o = {0, 0, 0, 0, 0};
      if (g0 + lane < nn) {
        np = v.pair_nbr[pi.nbr_begin + g0 + lane];
        const PairInfo& qn = v.pairs[np];
        nx = pi.x0 - qn.x0;                    // from the own patch to the neighbour's
        ny = pi.y0 - qn.y0;
        o = chunk_overlap(c0, c1, pi.w, nx, ny, qn.w, qn.h);
      }
      unsigned todo = __ballot_sync(0xffffffffu, o.begin < o.end);
      for (; todo; todo &= todo - 1) {
        const int g = __ffs(todo) - 1;
        const int bx = __shfl_sync(0xffffffffu, o.x, g), by = __shfl_sync(0xffffffffu, o.y, g);
        const int bw = __shfl_sync(0xffffffffu, o.w, g);
        const int b0 = __shfl_sync(0xffffffffu, o.begin, g);
        const int b1 = __shfl_sync(0xffffffffu, o.end, g);
        const int mx = __shfl_sync(0xffffffffu, nx, g), my = __shfl_sync(0xffffffffu, ny, g);
        stage_value(rec, v, __shfl_sync(0xffffffffu, np, g), lane, ne, nd);
        for_moments(rec, b0, b1, bw, bx + mx, by + my, lane, ne, nd,
                           [](int, int, int) { return 0; },
                           [&](int, int, int qx, int qy, float Es, float Vs) {
          const int q = (by + qy) * pi.w + bx + qx - c0;
          const float2 b = sum[q];
          sum[q] = make_float2(b.x + Es, b.y + Vs);
        });
      }
    }
    __syncwarp();
    for (int q = c0 + lane; q < c1; q += 32) v.bg[pi.bg_base + q] = sum[q - c0];
  }
}

// With a render cache (kOwn: with the plan's own renders of its neighbours)
// the neighbours' moments are gathered from it (the values the rendering would produce, added in the same order): the lane's
// eight pixels of the chunk stay in registers, and the neighbours' values
// come through asynchronous copies to shared memory (st: kBgCacheF floats of
// the warp), kBgStages - 1 neighbours ahead of the one being added, zeros
// where the pixel is not in the neighbour's patch.  Bound by memory latency:
// loads that a lane waits for, one neighbour or one pixel at a time, reach
// 1.6-1.9 TB/s (a Newton pass over 2,000 blended sources: 1.02 ms of
// preparation launches, 1.58 with a pixel's neighbours one after another).
__device__ __forceinline__ void copy_async8(unsigned dst, const void* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src),
               "r"(valid ? 8 : 0)
               : "memory");
}
template <bool kOwn>
__device__ __forceinline__ void background_cached(const PlanView& v, const Item& item,
                                                  const PairInfo& pi, float* st, int lane) {
  constexpr int kPix = kBgChunk / 32;
  const celeste_image& im = v.images[pi.image];
  const float2* stage = reinterpret_cast<const float2*>(st) + lane;
  const unsigned dst0 = (unsigned)__cvta_generic_to_shared(st) + lane * sizeof(float2);
  const int end = item.start + item.count;
  const int nn = pi.nbr_end - pi.nbr_begin;
  for (int c0 = item.start; c0 < end; c0 += kBgChunk) {
    const int c1 = min(c0 + kBgChunk, end);
    int x[kPix], y[kPix];
    float2 b[kPix];
    PixelWalk pw(c0 + lane, pi.w);
#pragma unroll
    for (int u = 0; u < kPix; ++u, pw.next(pi.w)) {
      const bool in = c0 + lane + 32 * u < c1;
      x[u] = in ? pw.qx : -(1 << 20);          // (outside every patch)
      y[u] = pw.qy;
      if (in) b[u] = make_float2(sky_checked(v, im, (float)(pi.x0 + pw.qx), (float)(pi.y0 + pw.qy)), 0.f);
    }
    const int r0 = c0 / pi.w, r1 = (c1 - 1) / pi.w + 1;   // the chunk's rows
    for (int g0 = 0; g0 < nn; g0 += 32) {
      // up to 32 neighbours, one in each lane
      int nx = 0, ny = 0, nw = 0, nh = 0;
      int64_t off = 0;
      if (g0 + lane < nn) {
        const PairInfo& qn = v.pairs[v.pair_nbr[pi.nbr_begin + g0 + lane]];
        nx = pi.x0 - qn.x0;                    // from the own patch to the neighbour's
        ny = pi.y0 - qn.y0;
        nw = qn.w;
        nh = qn.h;
        off = kOwn ? qn.bg_base : v.patches[qn.patch].pool_offset + cache_base(v, qn.source);
      }
      unsigned todo = __ballot_sync(0xffffffffu, min(r1, nh - ny) > max(r0, -ny) &&
                                                     min(pi.w, nw - nx) > max(0, -nx));
      const int cnt = __popc(todo);
      for (int k = 0; k < cnt + kBgStages - 1; ++k) {
        if (k < cnt) {
          const int g = __ffs(todo) - 1;
          todo &= todo - 1;
          const int mx = __shfl_sync(0xffffffffu, nx, g), my = __shfl_sync(0xffffffffu, ny, g);
          const int mw = __shfl_sync(0xffffffffu, nw, g), mh = __shfl_sync(0xffffffffu, nh, g);
          const float2* src = (kOwn ? v.nbr_render : v.cache) + __shfl_sync(0xffffffffu, off, g);
          const unsigned dst = dst0 + (k % kBgStages) * (kBgChunk * sizeof(float2));
#pragma unroll
          for (int u = 0; u < kPix; ++u) {
            const int lx = x[u] + mx, ly = y[u] + my;
            const bool in = (unsigned)lx < (unsigned)mw && (unsigned)ly < (unsigned)mh;
            copy_async8(dst + u * 32 * sizeof(float2), src + (in ? ly * mw + lx : 0), in);
          }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (k >= kBgStages - 1) {
          // each lane reads only what it copied itself
          asm volatile("cp.async.wait_group %0;" ::"n"(kBgStages - 1) : "memory");
          const float2* c = stage + ((k + 1) % kBgStages) * kBgChunk;
#pragma unroll
          for (int u = 0; u < kPix; ++u) {
            const float2 a = c[32 * u];
            b[u].x += a.x;
            b[u].y += a.y;
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kPix; ++u)
      if (c0 + lane + 32 * u < c1) v.bg[pi.bg_base + c0 + lane + 32 * u] = b[u];
  }
}

// Unit u of the backgrounds: its share of item u / split, whole lines of a warp
// (empty: count <= 0).
__device__ __forceinline__ Item item_share(const PlanView& v, int u, int split) {
  const int k = u / split;
  Item item = v.items[k];
  const int part = (item.count + 32 * split - 1) / (32 * split) * 32;
  const int skip = (u - k * split) * part;
  item.start += skip;
  item.count = min(part, item.count - skip);
  return item;
}

// Backgrounds of a plan without neighbours: the sky alone, as many warps as an
// SM takes (the log-likelihood of 600 sources in 2,400 items of 64 pixels:
// this launch 7.8 us, the rendering kernel 15.6).
__global__ void __launch_bounds__(128) sky_kernel(PlanView v, int split) {
  const int nwarps = gridDim.x * (blockDim.x >> 5);
  const int lane = threadIdx.x & 31;
  const int n = v.n_items * split;
  for (int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < n; u += nwarps) {
    const Item item = item_share(v, u, split);
    const PairInfo& pi = v.pairs[item.pair];
    if (item.count <= 0 || !v.active[pi.slot]) continue;
    const celeste_image& im = v.images[pi.image];
    const int end = item.start + item.count, w = pi.w, x0 = pi.x0, y0 = pi.y0;
    float2* bg = v.bg + pi.bg_base;
    PixelWalk pw(item.start + lane, w);
    for (int q = item.start + lane; q < end; q += 32, pw.next(w))
      bg[q] = make_float2(sky_checked(v, im, (float)(x0 + pw.qx), (float)(y0 + pw.qy)), 0.f);
  }
}

// Five blocks per SM (102 registers): 5-18 % faster than eight at 64.  split:
// the units of work that an item makes.
template <bool kQueue>
__global__ void __launch_bounds__(128, 5) background_kernel(PlanView v, int ne, int nd,
                                                            int split) {
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  float* rec = smem + wib * kBgWarpF;
  WarpQueue wq(kQueue ? v.work_ctr : nullptr);
  for (; wq.it < v.n_items * split; wq.advance()) {
    wq.ask(lane);
    const Item item = item_share(v, wq.it, split);
    const PairInfo pi = v.pairs[item.pair];
    if (item.count <= 0 || !v.active[pi.slot]) continue;
    background_rendered(v, item, pi, rec, lane, ne, nd);
  }
  wq.done(lane);
}

template <bool kOwn>
__global__ void __launch_bounds__(128) background_cached_kernel(PlanView v) {
  extern __shared__ float4 smem4[];
  const int lane = threadIdx.x & 31;
  float* st = reinterpret_cast<float*>(smem4) + (threadIdx.x >> 5) * kBgCacheF;
  const int nwarps = gridDim.x * (blockDim.x >> 5);
  for (int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < v.n_items; it += nwarps) {
    const Item item = v.items[it];
    const PairInfo pi = v.pairs[item.pair];
    if (v.active[pi.slot]) background_cached<kOwn>(v, item, pi, st, lane);
  }
}

// The start of an evaluation or of a Newton iteration of a colour class with
// a render cache, one warp per unit of work: the active set (a warp per 32
// slots; from the sources' status, every slot if that is null), the records
// of pairs [0, n_setup) at theta, and the background of every item of an
// active slot (the cache supplies the neighbours, so the own records are all
// it needs).
__global__ void __launch_bounds__(128) prepare_kernel(PlanView v, const ModelDev* __restrict__ model,
                                                      const int32_t* __restrict__ status,
                                                      int n_setup) {
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  float* rec = smem + wib * kBgCacheF;
  const int n_mark = (v.n + 31) / 32;
  const int units = n_mark + n_setup + v.n_items;
  // grid stride: its units are short, so a queue's claim would not return
  // before the next unit (measured 11 % slower)
  const int nwarps = gridDim.x * (blockDim.x >> 5);
  for (int u = blockIdx.x * (blockDim.x >> 5) + wib; u < units; u += nwarps) {
    if (u < n_mark) {
      const int j = 32 * u + lane;
      if (j < v.n) v.active[j] = status ? active_of(status[v.src_ids[j]]) : 1;
    } else if (u < n_mark + n_setup) {
      setup_pair(v, model, u - n_mark, false, rec, rec + 32, lane);
    } else {
      const Item item = v.items[u - n_mark - n_setup];
      const PairInfo pi = v.pairs[item.pair];
      if (status && !active_of(status[pi.source])) continue;
      background_cached<false>(v, item, pi, rec, lane);
    }
  }
}

// The loop of the render kernels: f(item, pair info) for every item.
template <bool kQueue, class F>
__device__ __forceinline__ void for_items(const PlanView& v, const Item* __restrict__ items, int n,
                                          int lane, F&& f) {
  WarpQueue wq(kQueue ? v.work_ctr : nullptr);
  for (; wq.it < n; wq.advance()) {
    wq.ask(lane);
    const Item item = items[wq.it];
    f(item, v.pairs[item.pair]);
  }
  wq.done(lane);
}

// Moments of the plan's neighbour pairs over their whole patches, once each,
// for the backgrounds to gather (into v.nbr_render); those that no active slot
// uses are passed by.  Bound by FP32 issue like
// the other renders; one pass over the patches instead of one an overlap
// (300 blended sources: render and gather 276 us, overlaps 750).
template <bool kQueue>
__global__ void __launch_bounds__(128, 8) render_neighbours_kernel(PlanView v, int ne, int nd) {
  extern __shared__ float4 smem4[];
  const int lane = threadIdx.x & 31;
  float* rec = reinterpret_cast<float*>(smem4) + (threadIdx.x >> 5) * kValRecF;
  for_items<kQueue>(v, v.nbr_items, v.n_nbr_items, lane, [&](const Item& item, const PairInfo& pi) {
    bool used = false;                       // by an active slot
    for (int k = pi.nbr_begin; k < pi.nbr_end && !used; k += 32)
      used = __any_sync(0xffffffffu, k + lane < pi.nbr_end && v.active[v.pair_nbr[k + lane]]);
    if (!used) return;
    float2* out = v.nbr_render + pi.bg_base;
    stage_value(rec, v, item.pair, lane, ne, nd);
    for_moments(rec, item.start, item.start + item.count, pi.w, 0, 0, lane, ne, nd,
                [](int, int, int) { return 0; }, [&](int, int q, int, int, float Es, float Vs) {
      out[q] = make_float2(Es, Vs);
    });
  });
}

// Own E_s and V_s of every plan pair, scattered to the caller's pool layout.
template <bool kQueue>
__global__ void __launch_bounds__(128, 8) render_kernel(PlanView v, int ne, int nd, float* E_out,
                                                        float* V_out,
                                                        const celeste_patch* __restrict__ patches) {
  extern __shared__ float4 smem4[];
  const int lane = threadIdx.x & 31;
  float* rec = reinterpret_cast<float*>(smem4) + (threadIdx.x >> 5) * kValRecF;
  for_items<kQueue>(v, v.items, v.n_items, lane, [&](const Item& item, const PairInfo& pi) {
    const int64_t off = patches[pi.patch].pool_offset;
    stage_value(rec, v, item.pair, lane, ne, nd);
    for_moments(rec, item.start, item.start + item.count, pi.w, 0, 0, lane, ne, nd,
                       [](int, int, int) { return 0; }, [&](int, int q, int, int, float Es, float Vs) {
      if (E_out) E_out[off + q] = Es;
      if (V_out) V_out[off + q] = Vs;
    });
  });
}

// Own E_s and V_s of the plan's pairs into the problem's render cache.
template <bool kQueue>
__global__ void __launch_bounds__(128, 8) render_cache_kernel(PlanView v, int ne, int nd,
                                                              const int32_t* __restrict__ status) {
  extern __shared__ float4 smem4[];
  const int lane = threadIdx.x & 31;
  float* rec = reinterpret_cast<float*>(smem4) + (threadIdx.x >> 5) * kValRecF;
  for_items<kQueue>(v, v.items, v.n_items, lane, [&](const Item& item, const PairInfo& pi) {
    if (status && status[pi.source] != CELESTE_ST_ACCEPTED) return;
    float2* out = v.cache + cache_base(v, pi.source) + v.patches[pi.patch].pool_offset;
    stage_value(rec, v, item.pair, lane, ne, nd);
    for_moments(rec, item.start, item.start + item.count, pi.w, 0, 0, lane, ne, nd,
                       [](int, int, int) { return 0; }, [&](int, int q, int, int, float Es, float Vs) {
      out[q] = make_float2(Es, Vs);
    });
  });
}

// A copy: every lane loads up to eight pixels before it stores any, so that
// enough loads are in flight to approach the copy bandwidth.
__global__ void __launch_bounds__(128) commit_render_kernel(PlanView v,
                                                            const int32_t* __restrict__ status) {
  const int nwarps = gridDim.x * (blockDim.x >> 5);
  const int lane = threadIdx.x & 31;
  for (int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < v.n_items; it += nwarps) {
    const Item item = v.items[it];
    const PairInfo pi = v.pairs[item.pair];
    if (status[pi.source] != CELESTE_ST_ACCEPTED) continue;
    const float2* __restrict__ src = v.trial_render + pi.bg_base + item.start;
    float2* __restrict__ dst =
        v.cache + cache_base(v, pi.source) + v.patches[pi.patch].pool_offset + item.start;
    const int n = item.count;
    for (int q0 = lane; q0 < n; q0 += 8 * 32) {
      float2 r[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (q0 + 32 * u < n) r[u] = __ldcs(src + q0 + 32 * u);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (q0 + 32 * u < n) dst[q0 + 32 * u] = r[u];
    }
  }
}

// Adds the plan's own moments into per-image buffers in the pixel-pool
// layout.  Plain read-modify-write: sources of one colour class never share
// a pixel, and classes are launched one after another.
template <bool kQueue>
__global__ void __launch_bounds__(128, 8) accumulate_kernel(PlanView v, int ne, int nd, float* Eimg,
                                                            float* Vimg) {
  extern __shared__ float4 smem4[];
  const int lane = threadIdx.x & 31;
  float* rec = reinterpret_cast<float*>(smem4) + (threadIdx.x >> 5) * kValRecF;
  for_items<kQueue>(v, v.items, v.n_items, lane, [&](const Item& item, const PairInfo& pi) {
    stage_value(rec, v, item.pair, lane, ne, nd);
    for_moments(rec, item.start, item.start + item.count, pi.w, 0, 0, lane, ne, nd,
                       [](int, int, int) { return 0; }, [&](int, int, int qx, int qy, float Es, float Vs) {
      const int64_t m = pi.pix_base + (int64_t)qy * pi.stride + qx;
      Eimg[m] += Es;
      Vimg[m] += Vs;
    });
  });
}

// Pixel term -E + x (log E - V / (2 E^2)) (Eq. eq:log_p_last, without
// log x!) over every pixel of image blockIdx.y, with E = sky + Eimg and
// V = Vimg; compensated FP32 sums per thread, FP64 across threads; one
// partial per block in parts[blockIdx.y * gridDim.x + blockIdx.x].  Four
// pixels' loads at a time and no division per pixel: 73 us for 15.2 M pixels
// (106 with a 64-bit division and one pixel at a time; the bytes take 27).
constexpr int kFieldBatch = 4;
__global__ void __launch_bounds__(256) field_term_kernel(const celeste_image* __restrict__ images,
                                                         const float* __restrict__ pixels,
                                                         const float* __restrict__ sky,
                                                         const float* __restrict__ Eimg,
                                                         const float* __restrict__ Vimg,
                                                         unsigned int* err, double* parts) {
  const celeste_image& im = images[blockIdx.y];
  const int w = im.width, stride = gridDim.x * blockDim.x;
  const int64_t n = (int64_t)im.height * w;
  const int64_t f0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  float s = 0.f, c = 0.f;
  // kFieldBatch of the thread's pixels at a time: their loads together, then
  // the terms in order.  Pixel coordinates step without a division.
  int x = (int)(f0 % w), y = (int)(f0 / w);
  const int ax = stride % w, ay = stride / w;
  for (int64_t f = f0; f < n; f += (int64_t)kFieldBatch * stride) {
    float e[kFieldBatch], V[kFieldBatch], cnt[kFieldBatch];
    int px[kFieldBatch], py[kFieldBatch];
#pragma unroll
    for (int u = 0; u < kFieldBatch; ++u) {
      px[u] = x;
      py[u] = y;
      if (f + (int64_t)u * stride < n) {
        const int64_t m = im.pix_offset + (int64_t)y * im.row_stride + x;
        e[u] = __ldcs(Eimg + m);
        V[u] = __ldcs(Vimg + m);
        cnt[u] = __ldcs(pixels + m);
      }
      x += ax;
      y += ay;
      if (x >= w) x -= w, ++y;
    }
#pragma unroll
    for (int u = 0; u < kFieldBatch; ++u) {
      if (f + (int64_t)u * stride < n) {
        const float sk = sky_value(im, sky, (float)px[u], (float)py[u]);
        if (!(sk > 0.f)) set_error(err, CELESTE_DERR_SKY);
        const float E = sk + e[u];
        const float r = __frcp_rn(E);
        const float t = fmaf(cnt[u], __logf(E) - 0.5f * V[u] * r * r, -E);
        const float yk = t - c;
        const float tk = s + yk;
        c = (tk - s) - yk;
        s = tk;
      }
    }
  }
  double d = (double)s - (double)c;
  d = warp_sum_d(d);
  __shared__ double red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = d;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
    parts[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = tot;
  }
}

// out[0] = sum parts - sum kl; out[1] = sum parts; out[2] = sum kl (fixed
// order, one block).
__global__ void __launch_bounds__(256) field_sum_kernel(const double* parts, int n_parts,
                                                        const double* kl, int n_kl, double* out) {
  __shared__ double red[2][256];
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < n_parts; i += blockDim.x) a += parts[i];
  for (int i = threadIdx.x; i < n_kl; i += blockDim.x) b += kl[i];
  red[0][threadIdx.x] = a;
  red[1][threadIdx.x] = b;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      red[0][threadIdx.x] += red[0][threadIdx.x + w];
      red[1][threadIdx.x] += red[1][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[1] = red[0][0];
    out[2] = red[1][0];
    out[0] = red[0][0] - red[1][0];
  }
}

// Backgrounds from the plan's pool to the caller's, eight loads in flight per
// lane (a copy: 167 us for 12.8 M pixels with one).
__global__ void __launch_bounds__(128) bg_scatter_kernel(PlanView v, float* bgE, float* bgV,
                                                         const celeste_patch* __restrict__ patches) {
  const int nwarps = gridDim.x * (blockDim.x >> 5);
  const int lane = threadIdx.x & 31;
  for (int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < v.n_items; it += nwarps) {
    const Item item = v.items[it];
    const PairInfo pi = v.pairs[item.pair];
    const int64_t off = patches[pi.patch].pool_offset + item.start;
    const float2* __restrict__ src = v.bg + pi.bg_base + item.start;
    for (int q0 = lane; q0 < item.count; q0 += 8 * 32) {
      float2 b[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (q0 + 32 * u < item.count) b[u] = __ldcs(src + q0 + 32 * u);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (q0 + 32 * u < item.count) {
          if (bgE) bgE[off + q0 + 32 * u] = b[u].x;
          if (bgV) bgV[off + q0 + 32 * u] = b[u].y;
        }
      }
    }
  }
}

static size_t smem_bytes(int wpb) { return (size_t)wpb * kValRecF * sizeof(float); }
static size_t smem_bytes_bg(int wpb) { return (size_t)wpb * kBgWarpF * sizeof(float); }
static size_t smem_bytes_cached(int wpb) { return (size_t)wpb * kBgCacheF * sizeof(float); }
static size_t smem_bytes_derivs(int wpb) { return (size_t)wpb * kDerivWarpF * sizeof(float); }
static size_t smem_bytes_grad(int wpb) { return (size_t)wpb * kDerivRecF * sizeof(float); }

constexpr int kWpb = 4;   // warps per block of the pixel kernels

// The derivative kernel's dynamic shared memory is close to the default 48 KB
// limit: raise the limit to what it uses.
static DeviceOnce g_derivs_attr;
using DerivsKernel = void (*)(PlanView, int, int);
static constexpr DerivsKernel kDerivsKernels[2][2] = {   // [queue][skip]
    {derivs_kernel<false, false>, derivs_kernel<false, true>},
    {derivs_kernel<true, false>, derivs_kernel<true, true>}};
static cudaError_t derivs_attr() {
  return g_derivs_attr.run([] {
    for (int k = 0; k < 4; ++k) {
      cudaError_t e = cudaFuncSetAttribute(kDerivsKernels[k / 2][k % 2],
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)smem_bytes_derivs(kWpb));
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  });
}

// Resident blocks per SM of each persistent pixel kernel, per device (0
// until measured on that device).
enum {
  kOccDerivs, kOccGrad, kOccValue, kOccDerivsQ, kOccGradQ, kOccValueQ, kOccBackground, kOccRender,
  kOccCommit, kOccPrepare, kOccCached, kOccKinds
};
static std::atomic<int> g_occ[kMaxDevices][kOccKinds] = {};
static DeviceOnce g_occ_once;

cudaError_t init_pixel_occupancy() {
  if (cudaError_t e = derivs_attr()) return e;
  return g_occ_once.run([] {
    const int dev = current_device();
    const size_t sm = smem_bytes(kWpb);
    int occ[kOccKinds] = {};
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &occ[kOccDerivs], kDerivsKernels[0][0], kWpb * 32, smem_bytes_derivs(kWpb));
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[kOccDerivsQ], kDerivsKernels[1][0],
                                                        kWpb * 32, smem_bytes_derivs(kWpb));
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[kOccGrad], grad_kernel<false>,
                                                        kWpb * 32, smem_bytes_grad(kWpb));
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[kOccGradQ], grad_kernel<true>,
                                                        kWpb * 32, smem_bytes_grad(kWpb));
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[kOccValue], value_kernel<false>,
                                                        kWpb * 32, sm);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[kOccValueQ], value_kernel<true>,
                                                        kWpb * 32, sm);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[kOccBackground],
                                                        background_kernel<true>, kWpb * 32,
                                                        smem_bytes_bg(kWpb));
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[kOccRender],
                                                        render_cache_kernel<true>, kWpb * 32,
                                                        sm);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[kOccCommit], commit_render_kernel,
                                                        kWpb * 32, 0);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[kOccPrepare], prepare_kernel,
                                                        kWpb * 32, smem_bytes_cached(kWpb));
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[kOccCached],
                                                        background_cached_kernel<true>,
                                                        kWpb * 32, smem_bytes_cached(kWpb));
    if (e == cudaSuccess)
      for (int k = 0; k < kOccKinds; ++k) g_occ[dev][k].store(occ[k], std::memory_order_relaxed);
    return e;
  });
}

// Persistent grid: SMs x (the tuning's blocks per SM, else the kernel's
// occupancy on the current device), no more blocks than the work needs.
static int grid_for(const Launch& L, int n_items, int wpb, int occ_kind = -1) {
  int per_sm = L.blocks_per_sm;
  if (per_sm <= 0) {
    const int occ =
        occ_kind >= 0 ? g_occ[current_device()][occ_kind].load(std::memory_order_relaxed) : 0;
    per_sm = occ > 0 ? occ : 3;
  }
  const int blocks = L.sm_count * per_sm;
  const int needed = (n_items + wpb - 1) / wpb;
  return blocks < needed ? blocks : (needed > 0 ? needed : 1);
}

// The work queue pays when a launch has many items per warp (its claims
// then balance the warps' finishing times); with few, the grid-stride form
// (fewer registers, no claims) is faster: from five items a warp in the
// derivative and value passes (batched field 12.57 -> 12.48 ms a pass for
// 2,000 sources against a line at eight; at three the sampler's value pass
// of 800 chains loses 4 %), from three in the gradient and rendering kernels
// (1,024 field sources: gradient 138 -> 129 us, backgrounds 50 -> 45).
constexpr int kQueueItems = 5, kQueueItemsRender = 3;
static bool use_queue(const PlanView& v, int n_items, int blocks, int per_warp) {
  return v.work_ctr && n_items >= per_warp * kWpb * blocks;
}

// Leaving out vanished pairs pays where pixels lie far from their source and
// the launch is bound by arithmetic: a mean patch of 45 x 45 pixels or more,
// and more items than warps on the GPU.  Batched field (2,000 sources, mean
// patch 2,700 pixels): 8.64 ms against 10.13; 1,200 field sources (mean
// patch 650): 0.615 against 0.604; one source of 101 x 101 pixels, which a
// few warps work on: 27.4 us against 26.9.
constexpr int kSkipArea = 2048;
static bool use_skip(const Launch& L, const PlanView& v) {
  return v.n_bg >= (int64_t)kSkipArea * v.n_own_pairs && v.n_items > 16 * L.sm_count;
}

// A launch over items of a value-only kernel, kernel(queue, grid) with queue
// a compile-time constant: with the work queue where the grid has many items
// per warp (occ_q: that form's occupancy).
template <class F>
static cudaError_t launch_items(const Launch& L, const PlanView& v, int n_items, int occ, int occ_q,
                                int per_warp, F&& kernel) {
  if (n_items == 0) return cudaSuccess;
  const int gq = grid_for(L, n_items, kWpb, occ_q);
  if (use_queue(v, n_items, gq, per_warp)) kernel(std::true_type(), gq);
  else kernel(std::false_type(), grid_for(L, n_items, kWpb, occ));
  return cudaGetLastError();
}

template <bool kOwn>
static cudaError_t launch_gather(const Launch& L, const PlanView& v) {
  if (v.n_items == 0) return cudaSuccess;
  background_cached_kernel<kOwn><<<grid_for(L, v.n_items, kWpb, kOccCached), kWpb * 32,
                                   smem_bytes_cached(kWpb), L.stream>>>(v);
  return cudaGetLastError();
}

cudaError_t launch_background(const Launch& L, const PlanView& v) {
  if (v.cache) return launch_gather<false>(L, v);
  if (v.nbr_render) {
    const cudaError_t e = launch_items(
        L, v, v.n_nbr_items, kOccRender, kOccRender, kQueueItemsRender, [&](auto q, int grid) {
          render_neighbours_kernel<decltype(q)::value>
              <<<grid, kWpb * 32, smem_bytes(kWpb), L.stream>>>(v, L.n_exp, L.n_dev);
        });
    return e == cudaSuccess ? launch_gather<true>(L, v) : e;
  }
  if (v.n_items == 0) return cudaSuccess;
  const int split = background_shares(v.n_bg, v.n_items, L.sm_count);
  if (v.n_pairs == v.n_own_pairs) {
    sky_kernel<<<grid_for(L, split * v.n_items, kWpb, kOccCommit), kWpb * 32, 0, L.stream>>>(v,
                                                                                            split);
    return cudaGetLastError();
  }
  return launch_items(L, v, split * v.n_items, kOccBackground, kOccBackground, kQueueItemsRender,
                      [&](auto q, int grid) {
    background_kernel<decltype(q)::value>
        <<<grid, kWpb * 32, smem_bytes_bg(kWpb), L.stream>>>(v, L.n_exp, L.n_dev, split);
  });
}

cudaError_t launch_pixels_derivs(const Launch& L, const PlanView& v) {
  if (v.n_items == 0) return cudaSuccess;
  if (block_per_item_derivs(v.n_bg, v.n_items, L.sm_count)) {
    derivs_coop_kernel<<<v.n_items, kCoopThreads, 0, L.stream>>>(v, L.n_exp, L.n_dev);
    return cudaGetLastError();
  }
  if (cudaError_t e = derivs_attr()) return e;
  const int gq = grid_for(L, v.n_items, kWpb, kOccDerivsQ);
  const bool queue = use_queue(v, v.n_items, gq, kQueueItems);
  const int grid = queue ? gq : grid_for(L, v.n_items, kWpb, kOccDerivs);
  kDerivsKernels[queue][use_skip(L, v)]<<<grid, kWpb * 32, smem_bytes_derivs(kWpb), L.stream>>>(
      v, L.n_exp, L.n_dev);
  return cudaGetLastError();
}

cudaError_t launch_pixels_grad(const Launch& L, const PlanView& v) {
  if (v.n_items == 0) return cudaSuccess;
  const int gq = grid_for(L, v.n_items, kWpb, kOccGradQ);
  if (use_queue(v, v.n_items, gq, kQueueItemsRender))
    grad_kernel<true><<<gq, kWpb * 32, smem_bytes_grad(kWpb), L.stream>>>(v, L.n_exp, L.n_dev);
  else
    grad_kernel<false><<<grid_for(L, v.n_items, kWpb, kOccGrad), kWpb * 32, smem_bytes_grad(kWpb),
                         L.stream>>>(v, L.n_exp, L.n_dev);
  return cudaGetLastError();
}

cudaError_t launch_pixels_value(const Launch& L, const PlanView& v, bool keep_render) {
  if (v.n_items == 0) return cudaSuccess;
  const int mode = !keep_render || !v.cache ? 0 : (v.cache_half ? 2 : 1);
  if (block_per_item_values(v.n_bg, v.n_items, L.sm_count)) {
    value_coop_kernel<<<v.n_items, kCoopThreads, 0, L.stream>>>(v, L.n_exp, L.n_dev, mode);
    return cudaGetLastError();
  }
  return launch_items(L, v, v.n_items, kOccValue, kOccValueQ, kQueueItems, [&](auto q, int grid) {
    value_kernel<decltype(q)::value>
        <<<grid, kWpb * 32, smem_bytes(kWpb), L.stream>>>(v, L.n_exp, L.n_dev, mode);
  });
}

cudaError_t launch_prepare(const Launch& L, const PlanView& v, const ModelDev* model,
                           const int32_t* status, int n_setup) {
  const int units = (v.n + 31) / 32 + n_setup + v.n_items;
  if (units == 0) return cudaSuccess;
  prepare_kernel<<<grid_for(L, units, kWpb, kOccPrepare), kWpb * 32, smem_bytes_cached(kWpb),
                   L.stream>>>(v, model, status, n_setup);
  return cudaGetLastError();
}

cudaError_t launch_commit_render(const Launch& L, const PlanView& v, const int32_t* status) {
  if (v.n_items == 0 || !v.cache || !v.trial_render) return cudaSuccess;
  commit_render_kernel<<<grid_for(L, v.n_items, kWpb, kOccCommit), kWpb * 32, 0, L.stream>>>(
      v, status);
  return cudaGetLastError();
}

cudaError_t launch_render(const Launch& L, const PlanView& v, float* E_out, float* V_out,
                          const celeste_patch* patches) {
  return launch_items(L, v, v.n_items, kOccRender, kOccRender, kQueueItemsRender, [&](auto q, int grid) {
    render_kernel<decltype(q)::value>
        <<<grid, kWpb * 32, smem_bytes(kWpb), L.stream>>>(v, L.n_exp, L.n_dev, E_out, V_out, patches);
  });
}

cudaError_t launch_render_cache(const Launch& L, const PlanView& v, const int32_t* status) {
  if (!v.cache) return cudaSuccess;
  return launch_items(L, v, v.n_items, kOccRender, kOccRender, kQueueItemsRender, [&](auto q, int grid) {
    render_cache_kernel<decltype(q)::value>
        <<<grid, kWpb * 32, smem_bytes(kWpb), L.stream>>>(v, L.n_exp, L.n_dev, status);
  });
}

cudaError_t launch_accumulate(const Launch& L, const PlanView& v, float* Eimg, float* Vimg) {
  return launch_items(L, v, v.n_items, kOccRender, kOccRender, kQueueItemsRender, [&](auto q, int grid) {
    accumulate_kernel<decltype(q)::value>
        <<<grid, kWpb * 32, smem_bytes(kWpb), L.stream>>>(v, L.n_exp, L.n_dev, Eimg, Vimg);
  });
}

cudaError_t launch_field_terms(const Launch& L, const celeste_image* images, int n_images,
                               int blocks_per_image, const float* pixels, const float* sky,
                               const float* Eimg, const float* Vimg, unsigned int* err,
                               double* parts) {
  if (n_images == 0) return cudaSuccess;
  field_term_kernel<<<dim3(blocks_per_image, n_images), 256, 0, L.stream>>>(images, pixels, sky,
                                                                            Eimg, Vimg, err, parts);
  return cudaGetLastError();
}

cudaError_t launch_field_sum(const Launch& L, const double* parts, int n_parts, const double* kl,
                             int n_kl, double* out) {
  field_sum_kernel<<<1, 256, 0, L.stream>>>(parts, n_parts, kl, n_kl, out);
  return cudaGetLastError();
}

cudaError_t launch_background_out(const Launch& L, const PlanView& v, float* bgE, float* bgV,
                                  const celeste_patch* patches) {
  if (v.n_items == 0) return cudaSuccess;
  bg_scatter_kernel<<<grid_for(L, v.n_items, kWpb, kOccCommit), kWpb * 32, 0, L.stream>>>(v, bgE, bgV,
                                                                                          patches);
  return cudaGetLastError();
}

}  // namespace celeste
