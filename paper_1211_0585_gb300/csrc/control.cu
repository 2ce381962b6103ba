// Device-resident iteration controller (Sect. 3 of the paper).
//
// Runs as the last kernel of every iteration: reduces the per-ring and per-m
// partial sums in a fixed order (bitwise reproducible), writes the
// iteration's record, and advances the schedule:
//   chi^2 = s^+ S^-1 s + (d - s)^+ N^-1 (d - s) of the iteration's input state;
//   while lambda > 1: after a chi^2 plateau (|chi2_k - chi2_{k-1}| below
//     plateau_eps * sigma_chi2, sigma_chi2 = sqrt(2 n_obs), both iterates of the
//     same level) double l_iter and lower lambda to C_{l_iter} / (tau Omega)
//     (clamped to >= 1; 1 once l_iter > lmax), band limit
//     lmax_SHT = min(lmax, l_iter + margin);
//   at lambda = 1 (band limit lmax): stop when the relative increment
//     ||s_k - s_{k-1}|| / ||s_k|| <= tol, or, if enabled, when
//     |Delta chi^2| < final_dchi2 * sigma_chi2 (the paper's rule, 1e-4).
// Keeping the controller on the device lets a whole block of iterations run
// as one CUDA graph with no host round trip.
#include <cuda_runtime.h>

#include "ctl.cuh"
#include "pdl.cuh"
#include "wf_internal.h"

namespace wfk {

// One CTA per controller (several maps' controllers share a launch). The launch
// is all latency on one SM: every thread's loads are independent and issued
// together; the FP64 pipe takes 16 cycles for a warp's addition, so the threads'
// sums meet in shared memory and one warp a quantity adds them (12 additions;
// by shuffles in every warp, 25, it took 7.0 us at Nside 16); thread 0
// advances a copy of the controller in shared memory instead of walking it in
// global memory field by field. 3.4 us at Nside 16, 6.7 us at Nside 512 (a tree
// over shared memory and the controller in global memory: 5.3 and 10.8).
constexpr int kCtlThreads = 256;
__global__ void __launch_bounds__(kCtlThreads) control_kernel(const __grid_constant__ CtlMaps Maps, int R, int lmax) {
  __shared__ double sh[5][kCtlThreads], tot[5];
  __shared__ Ctl live;
  const CtlMap &M = Maps.m[blockIdx.x];
  static_assert(sizeof(Ctl) % 4 == 0 && sizeof(Ctl) / 4 <= kCtlThreads, "copied a word a thread");
  constexpr int kWords = sizeof(Ctl) / 4;
  pdl_wait();
  pdl_next();
  if (threadIdx.x < kWords) reinterpret_cast<int *>(&live)[threadIdx.x] = reinterpret_cast<const int *>(M.ctl)[threadIdx.x];
  double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};   // chi2_N, chi2_lambda_N, chi2_S, increment, norm
  const double2 *rp = reinterpret_cast<const double2 *>(M.ring_part);
#pragma unroll 4
  for (int i = threadIdx.x; i < R; i += kCtlThreads) {
    const double2 r = rp[i];
    v[0] += r.x;
    v[1] += r.y;
  }
#pragma unroll 4
  for (int i = threadIdx.x; i <= lmax; i += kCtlThreads) {
    v[2] += M.m_part[3 * i];
    v[3] += M.m_part[3 * i + 1];
    v[4] += M.m_part[3 * i + 2];
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) sh[q][threadIdx.x] = v[q];
  __syncthreads();
  if (live.done) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < 5) {
    double t = sh[warp][lane];
#pragma unroll
    for (int i = 1; i < kCtlThreads / 32; ++i) t += sh[warp][32 * i + lane];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) tot[warp] = t;
  }
  __syncthreads();
  if (warp) return;
  if (lane == 0) ctl_advance(&live, M.cl, tot[2], tot[0], tot[1], tot[3], tot[4], M.hist, M.hist_cap, nullptr);
  __syncwarp();
  for (int i = lane; i < kWords; i += 32) reinterpret_cast<int *>(M.ctl)[i] = reinterpret_cast<const int *>(&live)[i];
}

void launch_control(const CtlMap *maps, int n, int R, int lmax, cudaStream_t s) {
  for (int i0 = 0; i0 < n; i0 += kCtlMapsMax) {
    CtlMaps q{};
    const int k = n - i0 < kCtlMapsMax ? n - i0 : kCtlMapsMax;
    for (int i = 0; i < k; ++i) q.m[i] = maps[i0 + i];
    launch_pdl(control_kernel, k, kCtlThreads, 0, s, q, R, lmax);
  }
}

}  // namespace wfk
