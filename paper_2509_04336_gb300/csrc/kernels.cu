// kernels.cu -- precision dispatch of the kernel launchers (kernels_p{0,1,2}.cu).
#include "gwns_internal.h"

namespace gwns {

// The inputs of a stand-alone walk that the caller's arrays do not hold, in one launch: the task
// travels as the kernel's argument (a pageable host copy held the host for ~10 us a call), and
// the survivors are split into float pairs once here; the walk kernels otherwise convert two
// survivors of FP64 for every candidate step, 22 conversions and 22 subtractions on the FP64
// pipe, which kept that pipe 18 % busy in the float-float walk.
__global__ void walk_prepare_kernel(WalkTask T, WalkTask* task, int32_t* blk_task, int32_t* blk_local, float2* survf,
                                    int32_t* clear, size_t n_surv) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    *task = T;
    if (clear) clear[0] = clear[1] = 0;
  }
  if (i < (size_t)T.n) {
    blk_task[i] = 0;
    blk_local[i] = (int32_t)i;
  }
  if (i < n_surv) {
    const double v = T.surv[i];
    const float vh = __double2float_rn(v);
    survf[i] = make_float2(vh, __double2float_rn(v - (double)vh));
  }
}

cudaError_t launch_walk_prepare(const WalkTask& T, WalkTask* d_task, int32_t* d_blk_task, int32_t* d_blk_local,
                                float2* d_survf, int32_t* clear, size_t n_surv, cudaStream_t s) {
  const size_t n = n_surv > (size_t)T.n ? n_surv : (size_t)T.n;
  walk_prepare_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(T, d_task, d_blk_task, d_blk_local, d_survf, clear,
                                                                  n_surv);
  return cudaGetLastError();
}

template <int P>
cudaError_t launch_likelihood_p(int waveform, int n_det, const EventDev* d_ev, const double* d_theta, int n,
                                double* d_lnl, int32_t* d_status, cudaStream_t s);
template <int P>
cudaError_t launch_unit_likelihood_p(int waveform, int n_det, const EventDev* d_ev, const double* d_u, int n,
                                     double* d_lnl, cudaStream_t s);
template <int P>
cudaError_t launch_walk_p(int waveform, int n_det, const EventDev* d_evs, WalkTask* d_tasks,
                          const int32_t* d_blk_task, const int32_t* d_blk_local, int n_blocks, cudaStream_t s,
                          int extras, bool chain);
template <int P>
cudaError_t launch_hrss_p(int waveform, int n_det, const EventDev* d_evs, WalkTask* d_tasks,
                          const int32_t* d_blk_task, const int32_t* d_blk_local, int n_blocks, cudaStream_t s);

cudaError_t launch_likelihood(int precision, int waveform, int n_det, const EventDev* d_ev, const double* d_theta,
                              int n, double* d_lnl, int32_t* d_status, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (precision == 0) return launch_likelihood_p<0>(waveform, n_det, d_ev, d_theta, n, d_lnl, d_status, s);
  if (precision == 1) return launch_likelihood_p<1>(waveform, n_det, d_ev, d_theta, n, d_lnl, d_status, s);
  return launch_likelihood_p<2>(waveform, n_det, d_ev, d_theta, n, d_lnl, d_status, s);
}

cudaError_t launch_unit_likelihood(int precision, int waveform, int n_det, const EventDev* d_ev, const double* d_u,
                                   int n, double* d_lnl, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (precision == 0) return launch_unit_likelihood_p<0>(waveform, n_det, d_ev, d_u, n, d_lnl, s);
  if (precision == 1) return launch_unit_likelihood_p<1>(waveform, n_det, d_ev, d_u, n, d_lnl, s);
  return launch_unit_likelihood_p<2>(waveform, n_det, d_ev, d_u, n, d_lnl, s);
}

cudaError_t launch_walk(int precision, int waveform, int n_det, const EventDev* d_evs, WalkTask* d_tasks,
                        const int32_t* d_blk_task, const int32_t* d_blk_local, int n_blocks, cudaStream_t s,
                        int extras, bool chain) {
  if (n_blocks <= 0) return cudaSuccess;
  if (precision == 0)
    return launch_walk_p<0>(waveform, n_det, d_evs, d_tasks, d_blk_task, d_blk_local, n_blocks, s, extras, chain);
  if (precision == 1)
    return launch_walk_p<1>(waveform, n_det, d_evs, d_tasks, d_blk_task, d_blk_local, n_blocks, s, extras, chain);
  return launch_walk_p<2>(waveform, n_det, d_evs, d_tasks, d_blk_task, d_blk_local, n_blocks, s, extras, chain);
}

cudaError_t launch_hrss(int precision, int waveform, int n_det, const EventDev* d_evs, WalkTask* d_tasks,
                        const int32_t* d_blk_task, const int32_t* d_blk_local, int n_blocks, cudaStream_t s) {
  if (n_blocks <= 0) return cudaSuccess;
  if (precision == 0) return launch_hrss_p<0>(waveform, n_det, d_evs, d_tasks, d_blk_task, d_blk_local, n_blocks, s);
  if (precision == 1) return launch_hrss_p<1>(waveform, n_det, d_evs, d_tasks, d_blk_task, d_blk_local, n_blocks, s);
  return launch_hrss_p<2>(waveform, n_det, d_evs, d_tasks, d_blk_task, d_blk_local, n_blocks, s);
}

}  // namespace gwns
