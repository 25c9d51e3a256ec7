#pragma once
// Sweeps of the C-first order (Algorithm 2) that only read R (templates;
// instantiated and launched by did_cfirst.cu).
//
// In this order b is fixed while c_1..c_K are updated, and c while b_1..b_K
// are.  With R_s the residual at the start of the sweep (kept unchanged), and c_l, c_l'
// (b_l, b_l') the blocks before and after their updates,
//   C step   b_k^T R  = b_k^T R_s  + sum_{l<k} (b_k.b_l) (c_l - c_l')
//   B step   R c_k'^T = R_s c_k'^T + sum_l [ b_l (c_l.c_k') - b_l* (c_l'.c_k') ],  b_l* = b_l' for l < k, else b_l.
// So the contractions of R_s do not depend on the updates of the same step, and
// one pass over R_s serves KB of them: KB rows of dots in the C step, KB
// columns of partials in the B step.  A sweep reads R 2 K / KB times and
// forms it anew from X at its end, where the sweep kernel reads and writes it
// 2 K times.  KB = 4 where a thread's KB vectors fit its registers.
//
// What bounds it: the HBM read of R_s (figures in did_cfirst.cu).  The stream, the
// producer and the pairs of float32 are those of did_defer_kernel.cuh.  The
// pending terms nearly cancel the contractions in the first sweeps, so they
// and the sums across warps, units and CTAs are kept as pairs.
#include "did_defer_kernel.cuh"

namespace did {
namespace cfirst_impl {

using namespace defer_impl;

constexpr int kThreads = kWorkThreads + 32;     // 16 computing warps and the producer warp

struct CfArgs {
  const void* R;
  float* B;            // ld x K
  float* C;            // K x N
  float* Co;           // K x N: c_l before its update
  float* T;            // [2][N][KB][GS / 32] the warps' parts of b_k^T R_s, passes alternate
  float* P;            // [2][KB][npart][ld] partial rows, passes alternate
  df* Gp;              // [K (K + 1) / 2][grid] per-CTA sums b_k.b_l, l <= k, at k (k + 1) / 2 + l
  df* Xp;              // [2][K][2 KB][grid] per-CTA sums c_l.c_k' and c_l'.c_k' of a block's KB columns
  unsigned* work;      // unit counters of the passes
  Ctrl* ctrl;
  unsigned long long* degen;
  int64_t N;
  int ld, K, GS, NG, S;
  Units units;
  int nunits, dynamic, npart;
  unsigned bar0;       // grid barriers of this sweep before this launch
  int bar_extra;
  uint64_t timeout_ns;
};

struct CfSmem {
  size_t ring, bo, bn, sums, acc, meta, cx, bars, misc, total;
};
__host__ __device__ __forceinline__ CfSmem cf_smem(int ld, int K, int grid, int S, int CW, int KB, int elem, bool bstep) {
  CfSmem L;
  const int rpc = defer_rows(ld, grid), st = rpc | 1;
  size_t o = 0;
  L.ring = o; o += ((size_t)S * CW * ld * elem + 127) & ~(size_t)127;
  L.bo = o;   o += al16((size_t)K * st * 4);
  L.bn = o;   o += bstep ? al16((size_t)K * st * 4) : 0;
  L.sums = o; o += al16((size_t)(bstep ? 2 : 1) * KB * K * 8);
  L.acc = o;  o += bstep ? al16((size_t)KB * 4 * kWorkThreads * 8) : 0;
  L.meta = o; o += (size_t)S * 16;
  L.cx = o;   o += al16((size_t)S * CW * KB * 4);
  L.bars = o; o += (size_t)2 * S * 8;
  L.misc = o; o += 64;
  L.total = o;
  return L;
}

// Whether an earlier launch stopped or failed (the C step of this sweep included):
// nothing of this one runs then.  err may also be of this launch, set by a CTA
// ahead of this one; the CTAs that began then leave at their next wait.  One
// thread reads, so that a CTA's threads agree.
__device__ __forceinline__ bool launch_ended(const Ctrl* ctrl) {
  return __syncthreads_or(threadIdx.x == 0 && (ld_volatile(&ctrl->stopped) != 0 || ld_volatile(&ctrl->err) != 0)) != 0;
}

// What both kernels set up.
struct Cta {
  unsigned char* ring;
  float *bos, *bns, *cxs;
  df *sums, *acc;
  StageMeta* meta;
  uint64_t *full, *empty;
  volatile int* quit;
  int* s_ok;
};
__device__ __forceinline__ Cta cf_setup(unsigned char* smem, const CfSmem& L, int S, int warps) {
  Cta c;
  c.ring = smem + L.ring;
  c.bos = reinterpret_cast<float*>(smem + L.bo);
  c.bns = reinterpret_cast<float*>(smem + L.bn);
  c.sums = reinterpret_cast<df*>(smem + L.sums);
  c.acc = reinterpret_cast<df*>(smem + L.acc);
  c.meta = reinterpret_cast<StageMeta*>(smem + L.meta);
  c.cxs = reinterpret_cast<float*>(smem + L.cx);
  c.full = reinterpret_cast<uint64_t*>(smem + L.bars);
  c.empty = c.full + S;
  c.quit = reinterpret_cast<volatile int*>(smem + L.misc);
  c.s_ok = reinterpret_cast<int*>(smem + L.misc) + 1;
  if ((int)threadIdx.x < S) {
    mbar_init(c.full + threadIdx.x, 1);
    mbar_init(c.empty + threadIdx.x, warps);
  }
  if (threadIdx.x == 0) *c.quit = 0;
  fence_mbar_init();
  __syncthreads();
  return c;
}

#define DID_CF_GRID_SYNC()                                                                                      \
  do {                                                                                                          \
    ++nbar;                                                                                                     \
    if (!work_grid_sync(&a.ctrl->bar, nbar * (unsigned)G + (unsigned)a.bar_extra, err, tmo, sm.s_ok, sm.quit)) { \
      if (t == 0) *sm.quit = 1;                                                                                 \
      return;                                                                                                   \
    }                                                                                                           \
  } while (0)

// -------------------------------------------------------------------- C step
template <int NR, int CW, int KB, bool BF16>
__global__ void __launch_bounds__(kThreads, 1) cstep_kernel(CfArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  if (launch_ended(a.ctrl)) return;
  typedef Vec<BF16> V;
  typedef typename V::raw raw;
  constexpr int VR = V::kRows, VH = VR / 2, ELEM = BF16 ? 2 : 4;
  constexpr int NV = KB * CW;                     // dot products of a chunk
  const int G = gridDim.x, cta = blockIdx.x, t = threadIdx.x, w = t >> 5, lane = t & 31;
  const int ld = a.ld, K = a.K, S = a.S, NG = a.NG, GS = a.GS;
  const int64_t N = a.N;
  const CfSmem L = cf_smem(ld, K, G, S, CW, KB, ELEM, false);
  const Cta sm = cf_setup(smem, L, S, GS / 32);
  int* err = &a.ctrl->err;
  const uint64_t tmo = a.timeout_ns;
  const uint32_t colbytes = (uint32_t)ld * ELEM, stagebytes = (uint32_t)CW * colbytes;
  const int passes = (K + KB - 1) / KB;

  if (w == kWorkThreads / 32) {
    Stream p{a.R, N, colbytes, sm.ring, sm.meta, sm.cxs, CW, sm.full, sm.empty, S, NG, G, cta, a.units, a.nunits,
             a.dynamic, a.work, sm.quit, err, tmo};
    produce<CW, 1>(p, 0, passes, [](int, int) -> const float* { return nullptr; });
    return;
  }

  unsigned nbar = a.bar0;
  const int g = t / GS, lt = t - g * GS, W = GS >> 5, wg = lt >> 5;
  const int nvec = ld / VR;
  const bool last_ok = lt + (NR - 1) * GS < nvec;
  unsigned cst = (unsigned)g % (unsigned)S, cph = ((unsigned)g / (unsigned)S) & 1u;
  const int rpc = defer_rows(ld, G), rst = rpc | 1;
  const int r0 = cta * rpc, nrows = max(0, min(ld, r0 + rpc) - r0);
  int64_t jlo, jhi;
  if (a.dynamic) {
    jlo = N * cta / G;
    jhi = N * (cta + 1) / G;
  } else {
    unit_range(a.units, N, cta, jlo, jhi);
  }

  // b_k.b_l for every pair: this CTA's rows
  for (int i = t; i < K * nrows; i += kWorkThreads) {
    const int k = i / nrows, r = i - k * nrows;
    sm.bos[k * rst + r] = __ldcg(a.B + (size_t)k * ld + r0 + r);
  }
  work_sync();
  const int npairs = K * (K + 1) / 2;
  for (int e = t; e < npairs; e += kWorkThreads) {
    int k = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    while (k * (k + 1) / 2 > e) --k;
    while ((k + 1) * (k + 2) / 2 <= e) ++k;
    const int l = e - k * (k + 1) / 2;
    df q = df_zero();
    for (int r = 0; r < nrows; ++r) q = df_fma(sm.bos[k * rst + r], sm.bos[l * rst + r], q);
    __stcg(reinterpret_cast<float2*>(a.Gp + (size_t)e * G + cta), make_float2(q.h, q.l));
  }
  DID_CF_GRID_SYNC();

  for (int p = 0; p < passes; ++p) {
    const int k0 = p * KB, kb = min(KB, K - k0);
    float* T = a.T + (size_t)(p & 1) * N * KB * W;
    // b_k of this thread's rows for the block's k
    float2 bn[KB][NR][VH];
#pragma unroll
    for (int i = 0; i < KB; ++i)
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int q = lt + r * GS;
        const bool in = i < kb && (r < NR - 1 || last_ok);
#pragma unroll
        for (int e = 0; e < VR; e += 4) {
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (in) v = __ldcg(reinterpret_cast<const float4*>(a.B + (size_t)(k0 + i) * ld + (size_t)q * VR + e));
          bn[i][r][e / 2] = make_float2(v.x, v.y);
          bn[i][r][e / 2 + 1] = make_float2(v.z, v.w);
        }
      }
    while (true) {
      if (!stage_wait(sm.full + cst, cph, err, tmo)) {
        *sm.quit = 1;                              // the CTA leaves after this pass
        break;
      }
      const int64_t j = sm.meta[cst].j;
      const int n = sm.meta[cst].n;
      const unsigned st = cst;
      cst += (unsigned)NG;
      while (cst >= (unsigned)S) {
        cst -= (unsigned)S;
        cph ^= 1u;
      }
      if (n < 0) {
        __syncwarp();
        if (lane == 0) mbar_arrive(sm.empty + st);
        break;
      }
      const raw* col = reinterpret_cast<const raw*>(sm.ring + (size_t)st * stagebytes) + lt;
      float2 d[NV];
#pragma unroll
      for (int e = 0; e < NV; ++e) d[e] = make_float2(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < CW; ++c) {
        if (c < n) {
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            if (r < NR - 1 || last_ok) {
              float f[VR];
              V::unpack(col[(size_t)c * nvec + r * GS], f);
#pragma unroll
              for (int h = 0; h < VH; ++h) {
                const float2 f2 = make_float2(f[2 * h], f[2 * h + 1]);
#pragma unroll
                for (int i = 0; i < KB; ++i) d[c * KB + i] = __ffma2_rn(bn[i][r][h], f2, d[c * KB + i]);
              }
            }
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(sm.empty + st);
      float v[NV];
#pragma unroll
      for (int e = 0; e < NV; ++e) v[e] = d[e].x + d[e].y;
      int m = 16;
#pragma unroll
      for (int h = NV / 2; h >= 1; h >>= 1) {
        const bool up = (lane & m) != 0;
#pragma unroll
        for (int e = 0; e < h; ++e) {
          const float send = up ? v[e] : v[e + h], keep = up ? v[e + h] : v[e];
          v[e] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
        m >>= 1;
      }
#pragma unroll
      for (int mm = 16 / NV; mm >= 1; mm >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], mm);
      const int e = lane / (32 / NV), c = e / KB;
      if ((lane & (32 / NV - 1)) == 0 && c < n) __stcg(T + ((size_t)(j + c) * KB + e % KB) * W + wg, v[0]);
    }
    // b_k.b_l of the block (sums[i * K + l])
    for (int i = 0; i < kb; ++i)
      sum_over_ctas(a.Gp + (size_t)(k0 + i) * (k0 + i + 1) / 2 * G, k0 + i + 1, G, sm.sums + (size_t)i * K);
    if (a.dynamic) {
      DID_CF_GRID_SYNC();
    } else {
      __threadfence_block();
      work_sync();
      if (*sm.quit) return;
    }
    // own columns: c_k' for the block's k in turn
    for (int64_t j = jlo + t; j < jhi; j += kWorkThreads) {
      df q[KB];
#pragma unroll
      for (int i = 0; i < KB; ++i) {
        q[i] = df_zero();
        if (i < kb)
          for (int e = 0; e < W; ++e) df_acc(q[i], __ldcg(T + ((size_t)j * KB + i) * W + e));
      }
      for (int l0 = 0; l0 < k0; l0 += 4) {        // (k0 is a multiple of KB, not always of 4)
        float cp[4], co[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const bool in = l0 + e < k0;
          cp[e] = in ? __ldcg(a.C + (int64_t)(l0 + e) * N + j) : 0.f;
          co[e] = in ? __ldcg(a.Co + (int64_t)(l0 + e) * N + j) : 0.f;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int l = l0 + e < k0 ? l0 + e : 0;
#pragma unroll
          for (int i = 0; i < KB; ++i)
            if (i < kb) {
              const df gl = sm.sums[i * K + l];
              q[i] = df_fma(co[e], gl, q[i]);
              q[i] = df_fma(-cp[e], gl, q[i]);
            }
        }
      }
#pragma unroll
      for (int i = 0; i < KB; ++i) {
        if (i < kb) {
          const int k = k0 + i;
          const float c_old = __ldcg(a.C + (int64_t)k * N + j);
          const df bb = sm.sums[i * K + k];
          float c_new = c_old;
          if (bb.h > 0.f) {
            const df v = df_div(df_fma(c_old, bb, q[i]), bb);
            c_new = v.h > 0.f ? v.h : 0.f;
          }
          __stcg(a.C + (int64_t)k * N + j, c_new);
          __stcg(a.Co + (int64_t)k * N + j, c_old);
#pragma unroll
          for (int i2 = i + 1; i2 < KB; ++i2)
            if (i2 < kb) {
              const df gl = sm.sums[i2 * K + k];
              q[i2] = df_fma(c_old, gl, q[i2]);
              q[i2] = df_fma(-c_new, gl, q[i2]);
            }
        }
      }
    }
    if (cta == 0 && t < kb && !(sm.sums[t * K + k0 + t].h > 0.f)) atomicAdd(a.degen, 1ull);
    work_sync();                                  // sums are free again
  }
}

// -------------------------------------------------------------------- B step
template <int NR, int CW, int KB, bool BF16>
__global__ void __launch_bounds__(kThreads, 1) bstep_kernel(CfArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  if (launch_ended(a.ctrl)) return;
  typedef Vec<BF16> V;
  typedef typename V::raw raw;
  constexpr int VR = V::kRows, VH = VR / 2, ELEM = BF16 ? 2 : 4;
  constexpr int KC = KB < 4 ? KB : 4;             // columns of C' summed at a time (eight sums)
  const int G = gridDim.x, cta = blockIdx.x, t = threadIdx.x, w = t >> 5, lane = t & 31;
  const int ld = a.ld, K = a.K, S = a.S, NG = a.NG, GS = a.GS;
  const int64_t N = a.N;
  const CfSmem L = cf_smem(ld, K, G, S, CW, KB, ELEM, true);
  const Cta sm = cf_setup(smem, L, S, GS / 32);
  int* err = &a.ctrl->err;
  const uint64_t tmo = a.timeout_ns;
  const uint32_t colbytes = (uint32_t)ld * ELEM, stagebytes = (uint32_t)CW * colbytes;
  const int passes = (K + KB - 1) / KB;

  if (w == kWorkThreads / 32) {
    Stream p{a.R, N, colbytes, sm.ring, sm.meta, sm.cxs, CW * KB, sm.full, sm.empty, S, NG, G, cta, a.units, a.nunits,
             a.dynamic, a.work, sm.quit, err, tmo};
    produce<CW, KB>(p, 0, passes, [&](int q, int i) -> const float* {
      return q * KB + i < K ? a.C + (int64_t)(q * KB + i) * N : nullptr;
    });
    return;
  }

  unsigned nbar = a.bar0;
  const int g = t / GS, lt = t - g * GS;
  const int nvec = ld / VR;
  const bool last_ok = lt + (NR - 1) * GS < nvec;
  unsigned cst = (unsigned)g % (unsigned)S, cph = ((unsigned)g / (unsigned)S) & 1u;
  const int rpc = defer_rows(ld, G), rst = rpc | 1;
  const int r0 = cta * rpc, nrows = max(0, min(ld, r0 + rpc) - r0);
  const int64_t jlo = N * cta / G, jhi = N * (cta + 1) / G;
  for (int i = t; i < K * nrows; i += kWorkThreads) {
    const int k = i / nrows, r = i - k * nrows;
    const float b = __ldcg(a.B + (size_t)k * ld + r0 + r);
    sm.bos[k * rst + r] = b;
    sm.bns[k * rst + r] = b;
  }
  work_sync();

  for (int p = 0; p < passes; ++p) {
    const int k0 = p * KB, kb = min(KB, K - k0);
    df* Xp = a.Xp + (size_t)(p & 1) * K * 2 * KB * G;
    float* P = a.P + (size_t)(p & 1) * KB * a.npart * ld;
    // c_l.c_k' and c_l'.c_k' on the own columns: a warp per l
    for (int l = w; l < K; l += kWorkThreads / 32) {
#pragma unroll
      for (int i0 = 0; i0 < KB; i0 += KC) {
        df v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = df_zero();
#pragma unroll 2
        for (int64_t j = jlo + lane; j < jhi; j += 32) {
          const float co = __ldcg(a.Co + (int64_t)l * N + j), cp = __ldcg(a.C + (int64_t)l * N + j);
#pragma unroll
          for (int i = 0; i < KC; ++i) {
            const float c = i0 + i < kb ? __ldcg(a.C + (int64_t)(k0 + i0 + i) * N + j) : 0.f;
            v[2 * i] = df_fma(co, c, v[2 * i]);
            v[2 * i + 1] = df_fma(cp, c, v[2 * i + 1]);
          }
        }
        const df s = df_warp_sum8(v);
        if (lane < 2 * KC)
          __stcg(reinterpret_cast<float2*>(Xp + (size_t)(l * 2 * KB + 2 * i0 + lane) * G + cta), make_float2(s.h, s.l));
      }
    }
    // partials of R_s c_k'^T for the block's k
    {
      float2 q[KB][NR][VH];
#pragma unroll
      for (int i = 0; i < KB; ++i)
#pragma unroll
        for (int r = 0; r < NR; ++r)
#pragma unroll
          for (int h = 0; h < VH; ++h) q[i][r][h] = make_float2(0.f, 0.f);
      int cu = -1;
      auto flush = [&](int u) {
#pragma unroll
        for (int i = 0; i < KB; ++i) {
          float* Pu = P + ((size_t)i * a.npart + (size_t)(u * NG + g)) * ld;
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            const int x = lt + r * GS;
            if (i < kb && (r < NR - 1 || last_ok)) {
#pragma unroll
              for (int e = 0; e < VR; e += 4)
                __stcg(reinterpret_cast<float4*>(Pu + (size_t)x * VR + e),
                       make_float4(q[i][r][e / 2].x, q[i][r][e / 2].y, q[i][r][e / 2 + 1].x, q[i][r][e / 2 + 1].y));
            }
#pragma unroll
            for (int h = 0; h < VH; ++h) q[i][r][h] = make_float2(0.f, 0.f);
          }
        }
      };
      while (true) {
        if (!stage_wait(sm.full + cst, cph, err, tmo)) {
          *sm.quit = 1;
          break;
        }
        const int n = sm.meta[cst].n, u = sm.meta[cst].u;
        const unsigned st = cst;
        cst += (unsigned)NG;
        while (cst >= (unsigned)S) {
          cst -= (unsigned)S;
          cph ^= 1u;
        }
        if (n < 0) {
          __syncwarp();
          if (lane == 0) mbar_arrive(sm.empty + st);
          break;
        }
        if (u != cu) {
          if (cu >= 0) flush(cu);
          cu = u;
        }
        const raw* col = reinterpret_cast<const raw*>(sm.ring + (size_t)st * stagebytes) + lt;
#pragma unroll
        for (int c = 0; c < CW; ++c) {
          if (c < n) {
            float cx[KB];
#pragma unroll
            for (int i = 0; i < KB; ++i) cx[i] = sm.cxs[st * CW * KB + c * KB + i];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              if (r < NR - 1 || last_ok) {
                float f[VR];
                V::unpack(col[(size_t)c * nvec + r * GS], f);
#pragma unroll
                for (int h = 0; h < VH; ++h) {
                  const float2 f2 = make_float2(f[2 * h], f[2 * h + 1]);
#pragma unroll
                  for (int i = 0; i < KB; ++i) q[i][r][h] = __ffma2_rn(f2, make_float2(cx[i], cx[i]), q[i][r][h]);
                }
              }
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(sm.empty + st);
      }
      if (cu >= 0) flush(cu);
    }
    DID_CF_GRID_SYNC();
    // b_k' of the own rows.  sums[l * 2 KB + 2 i]: c_l.c_k', + 1: c_l'.c_k' (k = k0 + i)
    sum_over_ctas(Xp, K * 2 * KB, G, sm.sums);
    const int nq = rpc / 4, SU = kWorkThreads / nq;
    const int quad = t % nq, sub = t / nq;
    if (sub < SU && 4 * quad < nrows) {
      for (int i = 0; i < kb; ++i) {
        df q[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) q[e] = df_zero();
        const float* Pr = P + (size_t)i * a.npart * ld + r0 + 4 * quad;
        for (int gi0 = sub; gi0 < a.npart; gi0 += 8 * SU) {
          float4 v[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const int gi = gi0 + e * SU;
            v[e] = gi < a.npart ? __ldcg(reinterpret_cast<const float4*>(Pr + (size_t)gi * ld))
                                : make_float4(0.f, 0.f, 0.f, 0.f);
          }
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            df_acc(q[0], v[e].x);
            df_acc(q[1], v[e].y);
            df_acc(q[2], v[e].z);
            df_acc(q[3], v[e].w);
          }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) sm.acc[((size_t)i * SU + sub) * rpc + 4 * quad + e] = q[e];
      }
    }
    work_sync();
    const int LPR = rpc >= 32 ? 8 : 32;
    const int e0 = t & (LPR - 1);
    for (int row0 = 0; row0 < rpc; row0 += kWorkThreads / LPR) {
      const int row = row0 + t / LPR;
      const bool in = row < nrows;
      for (int i = 0; i < kb; ++i) {
        const int k = k0 + i;
        const df cc = sm.sums[k * 2 * KB + 2 * i + 1];
        df q = df_zero();
        if (in) {
          for (int e = e0; e < SU; e += LPR) q = df_add(q, sm.acc[((size_t)i * SU + e) * rpc + row]);
          for (int l = e0; l < K; l += LPR) {
            q = df_fma(sm.bos[l * rst + row], sm.sums[l * 2 * KB + 2 * i], q);
            q = df_fma(-sm.bns[l * rst + row], sm.sums[l * 2 * KB + 2 * i + 1], q);
          }
        }
        for (int m = LPR / 2; m >= 1; m >>= 1) q = df_add(q, df_shfl_xor(q, m));
        __syncwarp();
        if (in && e0 == 0) {
          const float b_old = sm.bos[k * rst + row];
          float b_new = b_old;
          if (cc.h > 0.f) {
            const df v = df_add(df{b_old, 0.f}, df_div(q, cc));
            b_new = v.h > 0.f ? v.h : 0.f;
          }
          sm.bns[k * rst + row] = b_new;
          __stcg(a.B + (size_t)k * ld + r0 + row, b_new);
          if (!(cc.h > 0.f) && r0 + row == 0) atomicAdd(a.degen, 1ull);
        }
        __syncwarp();                              // the row's lanes see b_k' in the next step
      }
    }
    work_sync();                                   // sums and acc are free again
  }
}
#undef DID_CF_GRID_SYNC

}  // namespace cfirst_impl
}  // namespace did
