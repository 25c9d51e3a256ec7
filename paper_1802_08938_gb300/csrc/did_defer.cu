// Planner and launcher of the read-only sweep (did_defer_kernel.cuh) and the
// small kernel that closes each of its sweeps.
//
// Measured on one GB300, a sweep with the refresh that ends it, against the
// sweep kernel that writes R (a plain read of 4 GB runs at 7.2 TB/s):
//   5000 x 200000, K = 50, float32       48.0 -> 30.6 ms (585 us a k: pass 545, 7.3 TB/s)
//   10000 x 100000, K = 100, bfloat16    75.1 -> 37.1 ms (365 us a k: pass 313, 6.4 TB/s)
//   784 x 70000, K = 16, float32         1.52 -> 0.90 ms (49 us a k: pass 31)
//   784 x 70000, K = 16, bfloat16        1.13 -> 0.70 ms (39 us a k: pass 20)
#include "did_defer_kernel.cuh"

#include <algorithm>

namespace did {

using namespace defer_impl;

namespace {

// Closes a sweep: f = 1/2 ||R||^2 from the refresh's per-CTA sums (a tree of
// fixed shape), the stopping rule, and the barrier and the unit counters cleared
// for the next launch.  After a sweep that failed it stops the later ones of the
// queue instead: their barrier and unit counters would begin where the
// failed one left them.  Nothing after a sweep that stopped.
constexpr int kCloseThreads = 128;
__global__ void defer_close_kernel(const double* part, int n, int stride, Ctrl* ctrl, unsigned* work, int nwork, double* trace,
                                   int stop_rule, double tol, double f_prev, double f0, int first) {
  __shared__ double sum[kCloseThreads];
  if (ctrl->stopped) return;
  if (ctrl->err) {
    __syncthreads();
    if (threadIdx.x == 0) ctrl->stopped = 1;
    return;
  }
  for (int i = threadIdx.x; i < nwork; i += blockDim.x) work[i] = 0u;
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += kCloseThreads) s += part[(size_t)i * stride];
  sum[threadIdx.x] = s;
  for (int h = kCloseThreads / 2; h > 0; h >>= 1) {
    __syncthreads();
    if ((int)threadIdx.x < h) sum[threadIdx.x] += sum[threadIdx.x + h];
  }
  if (threadIdx.x == 0) {
    const double f = 0.5 * sum[0], prev = first ? f_prev : trace[-1];
    *trace = f;
    ctrl->bar = 0u;
    ctrl->sweeps += 1;
    if (stop_rule == 1 && (f == 0.0 || (prev > 0.0 && fabs(prev - f) / prev < tol))) ctrl->stopped = 1;
    if (stop_rule == 2 && f <= tol * f0) ctrl->stopped = 1;
  }
}

}  // namespace

bool plan_defer(int ld, int64_t N, int K, bool bf16, int grid_override, DeferPlan* plan) {
  const int VR = bf16 ? 8 : 4, elem = bf16 ? 2 : 4;
  const int nvec = ld / VR;
  int dev = 0, optin = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (K > 128) return false;
  DeferPlan P{};
  P.grid = grid_override > 0 ? std::min(grid_override, sms) : sms;
  if (defer_rows(ld, P.grid) > kMaxRows) return false;
  // Threads of a column group: as few as hold a column in 16 rows each, so
  // that a warp's reduction is shared by much of a column and b_k', the
  // partials and a chunk stay in registers; 512 beyond that.
  P.GS = 32;
  while (P.GS < kWorkThreads && P.GS * 16 < ld) P.GS *= 2;
  P.NR = std::max(1, (nvec + P.GS - 1) / P.GS);
  if (P.NR > (bf16 ? 5 : kMaxNr)) return false;
  P.NG = kWorkThreads / P.GS;
  // Columns of a chunk: the widest (within the registers) of which the ring
  // holds two a group, and three at all.  The ring holds whole rounds of the groups: a stage
  // then always serves the same group, which waits for its chunks in turn (a
  // group a whole ring ahead of another's unfinished copy would take the
  // previous phase of its barrier for its own).
  const size_t budget = (size_t)optin - 1024;
  const int cw_max = P.NR > 4 ? 1 : (P.NR > (bf16 ? 2 : 3) ? 2 : kMaxCw);
  for (int CW = cw_max; CW >= 1 && P.S == 0; CW /= 2)
    for (int s = 96 / P.NG * P.NG; s >= std::max(3, 2 * P.NG); s -= P.NG)
      if (defer_smem(ld, K, P.grid, s, CW, elem).total <= budget) {
        P.CW = CW;
        P.S = s;
        break;
      }
  if (P.S == 0) return false;
  P.smem = defer_smem(ld, K, P.grid, P.S, P.CW, elem).total;
  P.func = bf16 ? defer_func_bf16(P.NR, P.CW) : defer_func_f32(P.NR, P.CW);
  if (!P.func) return false;
  cudaFuncAttributes fa{};
  int per_sm = 0;
  if (cudaFuncGetAttributes(&fa, P.func) != cudaSuccess ||
      cudaFuncSetAttribute(P.func, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, P.func, kDeferThreads, P.smem) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    return false;
  }
  // Column units of a CTA: three tiers of 60 / 30 / 10 % from a counter (see
  // did_sweep.cu: SMs do not get equal shares of the bandwidth) while the partial rows
  // written and read stay under 4 % of the residual's bytes (they stay in
  // L2), else one contiguous range a CTA.
  const int64_t TG = P.grid;
  const double frac = 8.0 * 4.0 * (double)TG * P.NG / ((double)N * elem);
  P.dynamic = N >= 64 * TG && frac <= 0.04 ? 1 : 0;
  Units U{};
  U.tg = TG;
  if (P.dynamic) {
    U.c0 = std::max<int64_t>(1, (int64_t)(0.6 * (double)N / (double)TG));
    U.n0 = std::min<int64_t>(N, U.c0 * TG);
    U.c1 = std::max<int64_t>(1, (int64_t)(0.3 * (double)N / (double)TG));
    U.n1 = std::min<int64_t>(N, U.n0 + U.c1 * TG);
    U.c2 = std::max<int64_t>(1, (N - U.n1 + 2 * TG - 1) / (2 * TG));
    P.nunits = (int)(2 * TG + (N - U.n1 + U.c2 - 1) / U.c2);
  } else {
    U.c0 = (N + TG - 1) / TG;
    U.n0 = U.n1 = N;
    U.c1 = U.c2 = 1;
    P.nunits = (int)TG;
  }
  P.units = U;
  P.npart = P.nunits * P.NG;
  *plan = P;
  return true;
}

size_t defer_pair_bytes(int K, int grid) { return sizeof(df) * (size_t)(2 * K + 2) * grid; }

cudaError_t launch_defer(const DeferPlan& plan, const DeferBuffers& b, int ld, int64_t N, int K, int npart_first,
                         int bar_extra, uint64_t timeout_ns, uint64_t* tstamp, int tstamp_cap, cudaStream_t s) {
  DeferArgs a{};
  a.R = b.R;
  a.B = b.B;
  a.Bo = b.Bo;
  a.C = b.C;
  a.Co = b.Co;
  a.T = b.T;
  a.corr = static_cast<df*>(b.corr);
  a.P = b.P;
  a.CC0 = b.CC0;
  a.Xp = static_cast<df*>(b.Xp);
  a.Yp = static_cast<df*>(b.Yp);
  a.work = b.work;
  a.ctrl = b.ctrl;
  a.degen = b.degen;
  a.N = N;
  a.ld = ld;
  a.K = K;
  a.GS = plan.GS;
  a.NG = plan.NG;
  a.S = plan.S;
  a.units = plan.units;
  a.nunits = plan.nunits;
  a.dynamic = plan.dynamic;
  a.npart = plan.npart;
  a.npart_first = npart_first;
  a.bar_extra = bar_extra;
  a.timeout_ns = timeout_ns;
  a.tstamp = tstamp;
  a.tstamp_cap = tstamp_cap;
  void* params[] = {&a};
  return cudaLaunchCooperativeKernel(plan.func, dim3(plan.grid), dim3(kDeferThreads), params, plan.smem, s);
}

cudaError_t launch_defer_close(const double* part, int n, int stride, Ctrl* ctrl, unsigned* work, int nwork, double* trace,
                               int stop_rule, double tol, double f_prev, double f0, bool first, cudaStream_t s) {
  defer_close_kernel<<<1, kCloseThreads, 0, s>>>(part, n, stride, ctrl, work, nwork, trace, stop_rule, tol, f_prev, f0,
                                       first ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace did
