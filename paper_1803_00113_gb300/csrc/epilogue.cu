// Per-source epilogue kernels (epilogue.cuh): reduce a source's tile sums,
// chain them to the 27 coordinates and add the KL term.
#include "device_once.h"
#include "epilogue.cuh"

namespace celeste {

template <int kMode>
struct EpiBlock {
  EpiShared<kMode> e;
  ModelDev::F32 f;
};
template <>
struct EpiBlock<0> {
  KlSmem e;
};

// use_trial: bit 0 evaluates theta_trial; bit 1 (value mode only) asks for
// the pixel part alone, without the KL (the log-likelihood of the source's
// point values relative to its absence).
template <int kMode>
__global__ void __launch_bounds__(kEpiThreads) epilogue_kernel(PlanView v,
                                                               const ModelDev* __restrict__ model,
                                                               double* elbo, double* elbo_rel,
                                                               double* grad_out, double* hess_out,
                                                               int use_trial) {
  extern __shared__ double smd[];
  EpiBlock<kMode>& S = *reinterpret_cast<EpiBlock<kMode>*>(smd);
  const int j = blockIdx.x, tid = threadIdx.x;
  if (!v.active[j]) return;
  const bool trial = (use_trial & 1) != 0, pixel_only = kMode == 0 && (use_trial & 2) != 0;
  const double* thd =
      trial ? v.theta_trial + (size_t)j * kTheta : v.theta + (size_t)v.src_ids[j] * kTheta;
  if (tid < kTheta) S.e.th[tid] = (real)thd[tid];
  // a value reads the model's constants once, where they are: staging them
  // first costs every block 1 us (600 and 1,216 sources: 29.6 against 27.7 us
  // a call)
  const ModelDev::F32* f = &model->f;
  if constexpr (kMode >= 1) {
    stage_model(S.f, model, tid, kEpiThreads);
    f = &S.f;
  }
  double rel, full;
  epilogue_source<kMode>(v, *f, model->n_color, S.e, j, tid, pixel_only, rel, full);
  if (tid == 0) {
    if (elbo) elbo[j] = full;
    if (elbo_rel) elbo_rel[j] = rel;
    // a non-finite value at a trial point is a rejected step, not an error
    if (!isfinite(full) && !trial) set_error(v.err, CELESTE_DERR_NONFINITE);
  }
  if constexpr (kMode >= 1) {
    int bad = 0;
    for (int e = tid; e < kTheta; e += kEpiThreads) {
      grad_out[(size_t)j * kTheta + e] = (double)S.e.gth[e];
      bad |= !isfinite(S.e.gth[e]);
    }
    for (int e = tid; e < (kMode == 2 ? kTheta * kTheta : 0); e += kEpiThreads) {
      hess_out[(size_t)j * kTheta * kTheta + e] = (double)S.e.Hth[e];
      bad |= !isfinite(S.e.Hth[e]);
    }
    if (__syncthreads_or(bad) && tid == 0) set_error(v.err, CELESTE_DERR_NONFINITE);
  }
}

// The dynamic shared memory limit of each epilogue kernel, once per device.
template <int kMode>
static cudaError_t set_smem_attr() {
  static DeviceOnce once;
  return once.run([] {
    return cudaFuncSetAttribute(epilogue_kernel<kMode>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(EpiBlock<kMode>));
  });
}

cudaError_t launch_epilogue(const Launch& L, const PlanView& v, const ModelDev* model,
                            double* elbo, double* elbo_rel, double* grad, double* hess) {
  if (v.n == 0) return cudaSuccess;
  if (cudaError_t e = set_smem_attr<2>()) return e;
  epilogue_kernel<2><<<v.n, kEpiThreads, sizeof(EpiBlock<2>), L.stream>>>(v, model, elbo, elbo_rel, grad,
                                                              hess, 0);
  return cudaGetLastError();
}

cudaError_t launch_epilogue_grad(const Launch& L, const PlanView& v, const ModelDev* model,
                                 double* elbo, double* elbo_rel, double* grad) {
  if (v.n == 0) return cudaSuccess;
  if (cudaError_t e = set_smem_attr<1>()) return e;
  epilogue_kernel<1><<<v.n, kEpiThreads, sizeof(EpiBlock<1>), L.stream>>>(v, model, elbo, elbo_rel, grad,
                                                              nullptr, 0);
  return cudaGetLastError();
}

cudaError_t launch_epilogue_value(const Launch& L, const PlanView& v, const ModelDev* model,
                                  double* elbo, double* elbo_rel, bool use_trial) {
  if (v.n == 0) return cudaSuccess;
  if (cudaError_t e = set_smem_attr<0>()) return e;
  epilogue_kernel<0><<<v.n, kEpiThreads, sizeof(EpiBlock<0>), L.stream>>>(v, model, elbo, elbo_rel, nullptr,
                                                              nullptr, use_trial ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_epilogue_loglik(const Launch& L, const PlanView& v, const ModelDev* model,
                                   double* out) {
  if (v.n == 0) return cudaSuccess;
  if (cudaError_t e = set_smem_attr<0>()) return e;
  epilogue_kernel<0><<<v.n, kEpiThreads, sizeof(EpiBlock<0>), L.stream>>>(v, model, nullptr, out,
                                                                      nullptr, nullptr, 2);
  return cudaGetLastError();
}

// KL_s of every slot's source at theta, into kl_out[source id] (for the
// full-field ELBO, Eq. elbo: the pixel sum minus the sum of the KL_s).
__global__ void kl_kernel(PlanView v, const ModelDev* __restrict__ model, double* kl_out) {
  __shared__ KlSmem S;
  const int j = blockIdx.x;
  const int lane = threadIdx.x;
  const int src = v.src_ids[j];
  if (lane < kTheta) S.th[lane] = (real)v.theta[(size_t)src * kTheta + lane];
  __syncwarp();
  kl_terms<0, false>(S.th, model->f, model->n_color, S, lane);
  __syncwarp();
  if (lane == 0) kl_out[src] = (double)S.kls[0];
}

cudaError_t launch_kl(const Launch& L, const PlanView& v, const ModelDev* model, double* kl_out) {
  if (v.n == 0) return cudaSuccess;
  kl_kernel<<<v.n, 32, 0, L.stream>>>(v, model, kl_out);
  return cudaGetLastError();
}

}  // namespace celeste
