// Planner and launcher of the C-first sweeps that only read R
// (did_cfirst_kernel.cuh).
//
// Measured on one GB300, a float32 sweep with the refresh that ends it, against
// the sweep kernel that reads and writes R 2 K times:
//   8165 x 18821, K = 20     9.63 -> 1.39 ms (10 passes of 85 us at 7.2 TB/s)
//   5000 x 200000, K = 50    124.9 -> 18.6 ms (26 passes of 555 us)
//   784 x 70000, K = 16      2.93 -> 0.57 ms
#include "did_cfirst_kernel.cuh"

#include <algorithm>

namespace did {

using namespace cfirst_impl;

namespace {

// Blocks of k a pass serves: as many as leave a thread's KB x 4 NR (8 NR) values at 64 or fewer.
constexpr int block_of(int NR, bool bf16) {
  return NR * (bf16 ? 8 : 4) <= 16 ? 4 : NR * (bf16 ? 8 : 4) <= 32 ? 2 : 1;
}
template <int NR, bool BF16>
void pick(int CW, const void** c, const void** b) {
  constexpr int KB = block_of(NR, BF16);
  if (CW == 2) {
    *c = reinterpret_cast<const void*>(&cstep_kernel<NR, 2, KB, BF16>);
    *b = reinterpret_cast<const void*>(&bstep_kernel<NR, 2, KB, BF16>);
  } else {
    *c = reinterpret_cast<const void*>(&cstep_kernel<NR, 1, KB, BF16>);
    *b = reinterpret_cast<const void*>(&bstep_kernel<NR, 1, KB, BF16>);
  }
}
void pick_funcs(bool bf16, int NR, int CW, const void** c, const void** b) {
  *c = *b = nullptr;
  if (bf16) {
    switch (NR) {
      case 1: return pick<1, true>(CW, c, b);
      case 2: return pick<2, true>(CW, c, b);
      case 3: return pick<3, true>(CW, c, b);
      case 4: return pick<4, true>(CW, c, b);
    }
    return;
  }
  switch (NR) {
    case 1: return pick<1, false>(CW, c, b);
    case 2: return pick<2, false>(CW, c, b);
    case 3: return pick<3, false>(CW, c, b);
    case 4: return pick<4, false>(CW, c, b);
    case 5: return pick<5, false>(CW, c, b);
    case 6: return pick<6, false>(CW, c, b);
  }
}

}  // namespace

bool plan_cfirst(int ld, int64_t N, int K, bool bf16, CfirstPlan* plan) {
  if (K > 128) return false;
  const int VR = bf16 ? 8 : 4, elem = bf16 ? 2 : 4;
  const int nvec = ld / VR;
  int dev = 0, optin = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  CfirstPlan P{};
  P.grid = sms;
  if (defer_rows(ld, P.grid) > kMaxRows) return false;
  P.GS = 32;
  while (P.GS < kWorkThreads && P.GS * 16 < ld) P.GS *= 2;
  const int NR = std::max(1, (nvec + P.GS - 1) / P.GS);
  if (NR > (bf16 ? 4 : 6)) return false;
  P.NG = kWorkThreads / P.GS;
  P.NR = NR;
  P.KB = block_of(NR, bf16);
  const size_t budget = (size_t)optin - 1024;
  int CW = 0;
  for (CW = 2; CW >= 1 && P.S == 0; --CW)
    for (int s = 96 / P.NG * P.NG; s >= std::max(3, 2 * P.NG); s -= P.NG)
      if (cf_smem(ld, K, P.grid, s, CW, P.KB, elem, true).total <= budget &&
          cf_smem(ld, K, P.grid, s, CW, P.KB, elem, false).total <= budget) {
        P.S = s;
        P.CW = CW;
        break;
      }
  if (P.S == 0) return false;
  pick_funcs(bf16, NR, P.CW, &P.cfunc, &P.bfunc);
  P.csmem = cf_smem(ld, K, P.grid, P.S, P.CW, P.KB, elem, false).total;
  P.bsmem = cf_smem(ld, K, P.grid, P.S, P.CW, P.KB, elem, true).total;
  const void* fs[2] = {P.cfunc, P.bfunc};
  const size_t ss[2] = {P.csmem, P.bsmem};
  for (int i = 0; i < 2; ++i) {
    cudaFuncAttributes fa{};
    int per_sm = 0;
    if (!fs[i] || cudaFuncGetAttributes(&fa, fs[i]) != cudaSuccess ||
        cudaFuncSetAttribute(fs[i], cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fs[i], kThreads, ss[i]) != cudaSuccess || per_sm < 1) {
      cudaGetLastError();
      return false;
    }
  }
  // Column units as in did_defer.cu; tiers are cut finer where a unit would
  // hold more than 400 columns, which keeps the partials' chains of additions short.
  const int64_t G = P.grid;
  const double frac = 8.0 * 4.0 * (double)G * P.NG * P.KB / ((double)N * elem);
  P.dynamic = N >= 64 * G && frac <= 0.15 ? 1 : 0;
  Units U{};
  if (P.dynamic) {
    const int64_t m = std::max<int64_t>(1, (int64_t)(0.6 * (double)N / (double)(G * 400 * P.NG)) + 1);
    const int64_t tg = G * m;
    U.tg = tg;
    U.c0 = std::max<int64_t>(1, (int64_t)(0.6 * (double)N / (double)tg));
    U.n0 = std::min<int64_t>(N, U.c0 * tg);
    U.c1 = std::max<int64_t>(1, (int64_t)(0.3 * (double)N / (double)tg));
    U.n1 = std::min<int64_t>(N, U.n0 + U.c1 * tg);
    U.c2 = std::max<int64_t>(1, (N - U.n1 + 2 * G - 1) / (2 * G));
    P.nunits = (int)(2 * tg + (N - U.n1 + U.c2 - 1) / U.c2);
  } else {
    U.tg = G;
    U.c0 = (N + G - 1) / G;
    U.n0 = U.n1 = N;
    U.c1 = U.c2 = 1;
    P.nunits = (int)G;
  }
  P.units = U;
  P.npart = P.nunits * P.NG;
  *plan = P;
  return true;
}

CfirstSizes cfirst_sizes(const CfirstPlan& p, int ld, int64_t N, int K) {
  CfirstSizes z;
  z.Co = (size_t)K * N * 4;
  z.T = (size_t)2 * N * p.KB * (p.GS / 32) * 4;
  z.P = (size_t)2 * p.KB * p.npart * ld * 4;
  z.Gp = sizeof(df) * (size_t)K * (K + 1) / 2 * p.grid;
  z.Xp = sizeof(df) * (size_t)2 * K * 2 * p.KB * p.grid;
  return z;
}

cudaError_t launch_cfirst(const CfirstPlan& plan, const CfirstBuffers& b, int ld, int64_t N, int K, int bar_extra,
                          uint64_t timeout_ns, cudaStream_t s) {
  CfArgs a{};
  a.R = b.R;
  a.B = b.B;
  a.C = b.C;
  a.Co = b.Co;
  a.T = b.T;
  a.P = b.P;
  a.Gp = static_cast<df*>(b.Gp);
  a.Xp = static_cast<df*>(b.Xp);
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
  a.bar0 = 0;
  a.bar_extra = bar_extra;
  a.timeout_ns = timeout_ns;
  void* params[] = {&a};
  cudaError_t e = cudaLaunchCooperativeKernel(plan.cfunc, dim3(plan.grid), dim3(kThreads), params, plan.csmem, s);
  if (e != cudaSuccess) return e;
  const int passes = (K + plan.KB - 1) / plan.KB;
  a.bar0 = 1u + (plan.dynamic ? (unsigned)passes : 0u);
  a.work = b.work + passes;
  return cudaLaunchCooperativeKernel(plan.bfunc, dim3(plan.grid), dim3(kThreads), params, plan.bsmem, s);
}

}  // namespace did
