// Per-(source, image) setup kernel: one warp per pair (setup.cuh), four
// pairs a block.
#include <math.h>

#include "setup.cuh"

namespace celeste {

constexpr int kSetupWarps = 4;

// mark: also sets the plan's active set, 1 every slot, 2 from the sources'
// status, a slot a thread.
__global__ void __launch_bounds__(32 * kSetupWarps) setup_kernel(PlanView v,
                                                                  const ModelDev* __restrict__ model,
                                                                  int first_pair, int n_pairs,
                                                                  int use_trial, int mark,
                                                                  const int32_t* __restrict__ status) {
  __shared__ float s_th[kSetupWarps][32];    // theta, FP32
  __shared__ float s_im[kSetupWarps][32];    // PSF [k][6], then wcs_A [4], calib
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int warp = blockIdx.x * kSetupWarps + wib;
  if (mark) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < v.n) v.active[j] = mark == 1 ? 1 : active_of(status[v.src_ids[j]]);
  }
  if (warp >= n_pairs) return;
  setup_pair(v, model, first_pair + warp, use_trial != 0, s_th[wib], s_im[wib], lane);
}

cudaError_t launch_setup(const Launch& L, const PlanView& v, const ModelDev* model,
                         int first_pair, int n_pairs, bool use_trial, int mark,
                         const int32_t* status) {
  const int marks = mark ? (v.n + 32 * kSetupWarps - 1) / (32 * kSetupWarps) : 0;
  const int pairs = (n_pairs + kSetupWarps - 1) / kSetupWarps;
  const int blocks = pairs > marks ? pairs : marks;
  if (blocks <= 0) return cudaSuccess;
  setup_kernel<<<blocks, 32 * kSetupWarps, 0, L.stream>>>(v, model, first_pair, n_pairs,
                                                          use_trial ? 1 : 0, mark, status);
  return cudaGetLastError();
}

}  // namespace celeste
