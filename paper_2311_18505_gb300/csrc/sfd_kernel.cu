// Persistent step kernel for the nonlinear planar stiff string
// (arXiv 2311.18505, Sec. 3.2 Eq. 4; excitations Sec. 3.3 Eqs. 5-6).
//
// One warp owns one string at a time and advances it for a whole job
// (thousands of steps) without leaving the SM.  Lane j owns the contiguous
// rows [j m, j m + m) of each grid (m odd, so a warp-wide shared-memory
// access to row j m + r is free of bank conflicts).  Up to 9 transverse rows
// per lane are held in registers (sfd_step_reg.cuh); larger grids keep every
// per-row array in the warp's shared-memory region (sfd_step_smem.cuh).
//
// The state is kept as (u^n, D = u^n - u^{n-1}) and each step solves for the
// acceleration a = u^{n+1} - 2u^n + u^{n-1} (run_job states the equations).
// g = u_l - u_{l-1} are interval differences, e the interval differences of
// the longitudinal field interpolated to the transverse nodes (P, linear),
// A the tridiagonal Theta + s0 - s1 d2 - d_+[ca g^2 d(.)] of the k^2-scaled
// transverse line of Eq. 4.  Solving for the small accelerations keeps FP32
// rounding proportional to the motion per step rather than the displacement.
//
// The coupled system is solved by block Gauss-Seidel: a transverse
// tridiagonal solve (partitioned Thomas per lane + parallel cyclic
// reduction over the 32 lane-boundary unknowns by shuffles) alternating with
// a longitudinal one (constant matrix, factored once per job) until the
// longitudinal acceleration stops changing.  When the longitudinal
// off-diagonal (sigma1 k / h_l^2) is tiny it is folded into the sweeps as a
// Jacobi update instead.  Hammer and bow forces are scalar eliminations
// through the unit-force response A^{-1} J solved alongside.
#include <cuda_runtime.h>

#include <mutex>

#include "sfd_step_smem.cuh"
#include "sfd_step_reg.cuh"

// One translation unit per transverse rows-per-lane class: compiled with
// -DSFD_MU=<1|3|5|7|9> for the register path, or without SFD_MU for the
// shared-memory path, so each kernel gets the registers its class needs.
#define SFD_CAT2(a, b) a##b
#define SFD_CAT(a, b) SFD_CAT2(a, b)
#ifdef SFD_MU
#define SFD_LAUNCHER SFD_CAT(launch_synth_reg, SFD_MU)
#define SFD_KERNEL SFD_CAT(synth_kernel_reg, SFD_MU)
#else
#define SFD_LAUNCHER launch_synth_smem
#define SFD_KERNEL synth_kernel_smem
#endif

namespace sfd {

// A job of a string that is already unstable: zeros, and nothing stepped.
// (Apart from step_string: the test in front of its time loop changed the
// loop's registers, 96 kHz bass strings 8.81 -> 9.03 ms a block of 1024.)
static __device__ __noinline__ void silent_job(const Job& job, int lane) {
  for (int64_t j = lane; j < job.n_samples; j += kWarp) job.out[j] = 0.f;
  if (lane == 0) job.desc->sc->next_out += job.n_samples;
  __syncwarp();
}

// Warps per CTA, one CTA per SM.  One row per lane fits 128 registers with
// little spilling, so 16 warps of it share an SM: 2432 equal strings take
// 2.4 us a step (plucked) and 3.5 us (bowed), against 3.9 and 5.4 us in two
// rounds of 8 warps at 255 registers.  Three rows per lane spill 200 bytes in
// the bowed instances at 168 registers (12 warps) and took 3.6 us a step
// instead of 2.9, more than the extra warps gain (4096-string batch 10.5 ms
// per 512 samples against 10.2), so they and the larger classes keep 8 warps.
#ifdef SFD_MU
constexpr int kMaxThreads = kWarp * (SFD_MU == 1 ? 16 : 8);
#else
constexpr int kMaxThreads = kWarp * 4;
#endif

// Which warp takes which string.  The host sorts a class's jobs by the
// instance of the step function they take and gives every CTA a segment of
// them of about equal cost (Job::seg); the CTA's `regions` warps start on
// the segment's first jobs and take the others as they finish, by a counter
// per segment, then those of segments still waiting.  So the warps of an SM
// step strings of one or two kinds: each instance's time loop is 10-25 KB of
// code, and with the kinds mixed on every SM (one queue for all CTAs) their
// instruction fetches missed the cache: 1000 mixed strings then took 14.3 us
// a step, in segments 8.8 us (7.0 us with every later change; one generic
// loop for every kind: 10.0 us).
//
// With group = 4 or 8 (register path only) the CTA's warps step one string at
// a time together: warp 0 takes the next job and passes it on through shared
// memory (jcell) behind the group's barrier.  The cells alternate so that one
// is rewritten only after every warp has passed the next barrier, i.e. after
// all have read it.
__global__ void __launch_bounds__(kMaxThreads, 1) SFD_KERNEL(const Job* __restrict__ jobs, int n_jobs,
                                                             int* __restrict__ counters, int warp_floats,
                                                             int queued, int group) {
  extern __shared__ float smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & (kWarp - 1);
#ifdef SFD_MU
  __shared__ __align__(16) float xcells[2048];   // [buffer][warp][lane][chg, mag, chx, mgx]
  __shared__ int jcell[2];                       // a group's job index, alternating
  const int npw = group;
#else
  const int npw = 1;
  (void)group;
#endif
  const int pi = warp / npw, pw = warp - pi * npw;
  const int regions = (blockDim.x >> 5) / npw;
  const int region = pi * warp_floats;
  const int n_ctas = gridDim.x;
  // the next job of segment v, or n_jobs; its first `regions` are taken as
  // the CTA starts, the others in the order of the segment's counter
  auto segment = [&](int v) { return v < n_ctas ? jobs[v].seg : n_jobs; };
  const int seg0 = segment(blockIdx.x), seg1 = segment(blockIdx.x + 1);
  auto take = [&](int v) {
    const int j = segment(v) + regions + atomicAdd(&counters[v], 1);
    return j < segment(v + 1) ? j : n_jobs;
  };
  auto next_job = [&](bool first) {
    if (first) return seg0 + pi < seg1 ? seg0 + pi : n_jobs;
    if (!queued) return n_jobs;   // every job began as its CTA started
    int j = n_jobs;
    if (lane == 0) j = take(blockIdx.x);
    j = __shfl_sync(SFD_FULL, j, 0);
    // this segment is empty: help the others, from the next one on
    for (int b = 0; j >= n_jobs && b < n_ctas; b += kWarp) {
      const int o = b + lane, v = o < n_ctas ? (blockIdx.x + 1 + o) % n_ctas : 0;
      const int seen = o < n_ctas ? *const_cast<volatile int*>(&counters[v]) : 0;
      unsigned left = __ballot_sync(SFD_FULL, o < n_ctas && segment(v) + regions + seen < segment(v + 1));
      while (left && j >= n_jobs) {
        const int src = __ffs(left) - 1;
        left &= left - 1;
        const int vv = __shfl_sync(SFD_FULL, v, src);
        if (lane == 0) j = take(vv);
        j = __shfl_sync(SFD_FULL, j, 0);
      }
    }
    return j;
  };
#ifdef SFD_MU
  int it = 0;
#endif
  for (bool first = true;; first = false) {
    int j = n_jobs;
    if (pw == 0) j = next_job(first);
#ifdef SFD_MU
    if (npw > 1) {
      if (pw == 0 && lane == 0) jcell[it & 1] = j;
      group_sync(npw);
      j = jcell[it & 1];
      ++it;
    }
#endif
    if (j >= n_jobs) break;
    if (jobs[j].desc->sc->status & kStUnstable) {
      if (pw == 0) silent_job(jobs[j], lane);
      continue;
    }
#ifdef SFD_MU
    run_job_reg<SFD_MU>(jobs[j], region, lane, pw, npw, xcells);
#else
    run_job(jobs[j], smem + region, lane);
#endif
  }
}

// The kernel's dynamic shared-memory limit is a process-wide attribute of
// the function on each device.  It is raised once per device to everything
// a block may opt into (minus the kernel's static shared memory) and never
// lowered, so launches from several threads or contexts cannot undo one
// another's setting between setting and launching; each launch still asks
// for only the bytes its strings need.
namespace {
constexpr int kMaxAttrDevices = 64;
std::mutex g_attr_mu;
bool g_attr_done[kMaxAttrDevices] = {};

cudaError_t raise_smem_limit() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxAttrDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_attr_mu);
  if (g_attr_done[dev]) return cudaSuccess;
  int optin = 0;
  e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, SFD_KERNEL);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(SFD_KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           optin - static_cast<int>(fa.sharedSizeBytes));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(SFD_KERNEL, cudaFuncAttributePreferredSharedMemoryCarveout, kSmemCarveout);
  if (e == cudaSuccess) g_attr_done[dev] = true;
  return e;
}
}  // namespace

// Host-side launcher of this class (C++ linkage, called by sfd_api.cu): CTA
// c steps its segment of the jobs, warps_per_cta / group of them at a time.
// With `queued` (some segment is longer than that) the CTAs take them by one
// counter each, cleared on the same stream before the kernel starts.  With
// group = 4 or 8 (register classes; warps_per_cta = group) each string gets
// the CTA's warps and one shared-memory region.  A priority other than 0 is
// the launch's own, whatever the stream's.
cudaError_t SFD_LAUNCHER(const Job* d_jobs, int n_jobs, int* d_counters, int warp_floats, int warps_per_cta,
                         int n_ctas, int queued, int group, int priority, cudaStream_t stream) {
#ifndef SFD_MU
  group = 1;
#endif
  if (group != 1 && group != 4 && group != 8) return cudaErrorInvalidValue;
  if (warps_per_cta < 1 || warps_per_cta * kWarp > kMaxThreads || (group > 1 && warps_per_cta != group))
    return cudaErrorInvalidValue;
  const int regions = warps_per_cta / group;
  const size_t smem = static_cast<size_t>(warp_floats) * regions * sizeof(float);
  cudaError_t e = raise_smem_limit();
  if (e != cudaSuccess) return e;
  if (queued) {
    e = cudaMemsetAsync(d_counters, 0, sizeof(int) * n_ctas, stream);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributePriority;
  attr.val.priority = priority;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_ctas);
  cfg.blockDim = dim3(warps_per_cta * kWarp);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = priority != 0 ? 1 : 0;
  e = cudaLaunchKernelEx(&cfg, SFD_KERNEL, d_jobs, n_jobs, d_counters, warp_floats, queued, group);
  const cudaError_t last = cudaGetLastError();   // (cleared, whatever the launch returned)
  return e != cudaSuccess ? e : last;
}

}  // namespace sfd
