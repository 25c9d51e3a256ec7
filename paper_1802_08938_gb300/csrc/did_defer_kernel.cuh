#pragma once
// Read-only sweep of the interleaved order (templates; instantiated by the
// did_defer_*.cu units, planned and launched by did_defer.cu).
//
// The sweep of did_sweep_kernel.cuh writes R for every k or every pair of k.
// Here R keeps the value R_s it had when the sweep began, and the changes of
// the blocks visited so far stay pending as vectors.  With b_l, c_l before and b_l',
// c_l' after their updates (l < k), the true residual is
//   R = R_s + sum_{l<k} (b_l c_l - b_l' c_l'),
// so the two contractions of step k (Section 2, HALS closed forms; Section 4.1,
// sol:b_i and up:c) are contractions of R_s plus scalars times vectors:
//   R c_k^T  = R_s c_k^T  + sum_l [ b_l (c_l.c_k) - b_l' (c_l'.c_k) ]
//   b_k'^T R = b_k'^T R_s + sum_l [ (b_k'.b_l) c_l - (b_k'.b_l') c_l' ]
// One pass over R_s per k gives b_k'^T R_s and the partials of R_s c_{k+1}^T
// from the same read; nothing is written.  After k = K the residual is formed anew
// from X (did_refresh_tc.cu, which also gives the objective and the partials
// for the next c_1).  A sweep so moves K passes of R plus the refresh (read X, write
// R), where writing R per pair of k moves 1.5 K and per k 2 K.
//
// What bounds it: the HBM read of R_s.  Measured at 5000 x 200000, K = 50
// and 10000 x 100000, K = 100 (bfloat16): see did_defer.cu.
//
// Per k, on a cooperative grid of one CTA per SM:
//   A   every CTA owns a slice of rows: R c_k^T from the partial rows and the
//       pending terms, b_k' (sol:b_i), and the slice's sums b_k'.b_l, b_k'.b_l'
//   --  grid barrier
//   S   stream R_s: 16 warps; a chunk of CW columns goes to a group of GS
//       threads, each thread holding NR 16-byte vectors of b_k' and of the
//       partials in registers.  A warp never waits for another: each stores
//       its rows' part of the dot product to T, and phase F adds the warps' parts.
//   B   beside S, on four warps of their own: for the CTA's own columns the
//       pending terms of c_k (a sum over l) and the sums c_l.c_{k+1},
//       c_l'.c_{k+1} (l < k).  On the 16 warps before S it took 23 us of each of
//       617 us at 5000 x 200000, K = 50.
//   --  grid barrier when column units come from a counter, else CTA barrier
//   F   own columns: c_k', and the sums for l = k
//   --  grid barrier
// A producer warp streams the columns by TMA bulk copies into one ring for
// the CTA and does not take part in the phases or barriers: R_s does not
// change, so the ring refills for the next pass while the phases run.  Its
// lanes each issue a chunk: one lane issuing them in turn took 290 ns a
// chunk, more than HBM takes for one of short columns.
//
// In the first sweeps R_s is much larger than R is later in the sweep, so the
// pending terms nearly cancel the contractions of R_s.  The scalars, the pending terms and
// the sums over warps, units and CTAs are therefore kept to about 45 bits: pairs
// of float32 (did_pair.cuh).  Errors against 64 bits come out below those of the
// kernel that writes R, whose partial rows are added in plain float32: B after three
// sweeps 0.5 to 0.8 times as far off on fourteen shapes (tests/test_gpu_defer.py
// prints both).
#include "did_internal.cuh"
#include "did_pair.cuh"

namespace did {
namespace defer_impl {

constexpr int kWorkThreads = 512;               // 16 warps that compute
constexpr int kSideThreads = 128;               // 4 warps for the pending terms (phase B)
constexpr int kDeferThreads = kWorkThreads + 32 + kSideThreads;   // and the producer warp
constexpr int kTiles = 4;                        // columns of a thread at a time in phases B and F
constexpr int kMaxCw = 4;                        // columns of a chunk (most)
constexpr int kMaxNr = 10;

// ------------------------------------------------------------- arguments
struct DeferArgs {
  const void* R;       // ld x N residual, constant in the launch (float or bfloat16)
  float* B;            // ld x K, rows >= M are zero
  float* Bo;           // ld x K: b_l before its update in this sweep
  float* C;            // K x N
  float* Co;           // K x N: c_l before its update in this sweep
  float* T;            // [N][GS / 32] the warps' parts of b_k'^T R_s
  df* corr;            // [N] pending terms of c_k
  float* P;            // partial rows of R_s c^T: [npart][ld] (the first step: npart_first rows)
  const double* CC0;   // [npart_first] partials of ||c_1||^2
  df* Xp;              // [2K + 1][grid] per-CTA sums: c_l.c, c_l'.c (l <= k), ||c||^2 with c = c_{k+1}
  df* Yp;              // [2K + 2][grid] per-CTA sums: b'.b_l, b'.b_l' (l < k), b'.b', b'.b_k
  unsigned* work;      // [K + 1] column-unit counters (pass k at k + 1), zeroed before the launch
  Ctrl* ctrl;
  unsigned long long* degen;
  int64_t N;
  int ld, K;
  int GS, NG;          // threads of a column group; groups of the CTA
  int S;               // ring stages (chunks of CW columns)
  Units units;         // column ranges of the CTA-level units
  int nunits, dynamic;
  int npart, npart_first;   // npart_first 0: no partials for c_1 yet, a first pass forms them
  int bar_extra;
  uint64_t timeout_ns;
  uint64_t* tstamp;    // phase stamps of this sweep (CTA 0), 4 per k, or null
  int tstamp_cap;
};

// Shared memory of a CTA (byte offsets; the same formula on host and device).
struct DeferSmem {
  size_t ring, bo, bn, xw, sums, accd, bk, meta, cx, bars, misc, total;
};
__host__ __device__ __forceinline__ size_t smax(size_t a, size_t b) { return a > b ? a : b; }
__host__ __device__ __forceinline__ size_t al16(size_t x) { return (x + 15) & ~(size_t)15; }
// Rows of a CTA's slice: a multiple of four, for 16-byte loads of the partial rows.
// A thread adds the partial rows of one quad of them, so a slice holds at
// most kMaxRows; the planners refuse longer ones (a grid of few CTAs).
constexpr int kMaxRows = 4 * kWorkThreads;
__host__ __device__ __forceinline__ int defer_rows(int ld, int grid) { return ((ld + grid - 1) / grid + 3) / 4 * 4; }
__host__ __device__ __forceinline__ DeferSmem defer_smem(int ld, int K, int grid, int S, int CW, int elem) {
  DeferSmem L;
  const int st = defer_rows(ld, grid) | 1;      // odd stride: a warp over l is free of bank conflicts
  size_t o = 0;
  L.ring = o; o += ((size_t)S * CW * ld * elem + 127) & ~(size_t)127;
  L.bo = o;   o += al16((size_t)K * st * 4);     // own rows of b_l
  L.bn = o;   o += al16((size_t)K * st * 4);     // own rows of b_l'
  // per-warp sums of phases B and F; phase A keeps its subsets' sums there
  L.xw = o;   o += al16(smax((size_t)20 * 2 * (K + 1) * 8, (size_t)4 * kWorkThreads * 8));
  L.sums = o; o += al16((size_t)(2 * K + 2) * 8);        // grid-wide sums
  L.accd = o; o += 2 * kWorkThreads * 8;         // sums of b_k'.b_l by parts of the rows
  L.bk = o;   o += al16((size_t)st * 4);         // own rows of b_k'
  L.meta = o; o += (size_t)S * 16;
  L.cx = o;   o += (size_t)S * kMaxCw * 4;
  L.bars = o; o += (size_t)2 * S * 8;
  L.misc = o; o += 64;
  L.total = o;
  return L;
}

struct StageMeta {
  int64_t j;   // first column
  int n;       // columns (0: none, only the unit counts; -1: end of the pass)
  int u;       // unit
};

__device__ __forceinline__ void work_sync() { named_bar(1, kWorkThreads); }
// The computing warps tell the side warps that the sums of phase A are there
// (barrier 2), the side warps that phase B is done (barrier 3): one half
// arrives, the other waits.
__device__ __forceinline__ void side_arrive(int id) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(kWorkThreads + kSideThreads) : "memory");
}
__device__ __forceinline__ void side_wait(int id) { named_bar(id, kWorkThreads + kSideThreads); }

// Grid barrier of the computing warps (see grid_sync): release add, acquire
// poll without back-off; the limit is read every 64 polls.  A CTA one of whose
// threads gave up waiting for a stage (*quit) does not arrive, so no CTA goes
// on with its partial sums.
__device__ __forceinline__ bool work_grid_sync(unsigned* bar, unsigned target, int* err, uint64_t timeout_ns,
                                               int* s_ok, volatile int* quit) {
  work_sync();
  if (*quit) return false;
  if (threadIdx.x == 0) {
    int ok = 1;
    __threadfence();
    atomicAdd(bar, 1u);
    uint64_t t0 = 0;
    for (unsigned i = 0; (int)(ld_acquire_gpu(bar) - target) < 0; ++i) {
      if ((i & 63u) == 63u) {
        const uint64_t t = globaltimer_ns();
        if (t0 == 0) t0 = t;
        if (ld_volatile(err) != 0) { ok = 0; break; }
        if (t - t0 > timeout_ns || i > (1u << 28)) {
          atomicCAS(err, 0, kDevErrTimeout);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
    *s_ok = ok;
  }
  work_sync();
  return *s_ok != 0;
}

// Wait of a whole warp for phase `parity` of a stage, bounded by the limit
// (looked at every 64 polls: %globaltimer is slow to read).  The lanes agree on the
// result, as what follows shuffles among all of them.
__device__ __forceinline__ bool stage_wait(uint64_t* b, uint32_t parity, int* err, uint64_t timeout_ns) {
  if (__all_sync(0xffffffffu, mbar_try_wait(b, parity))) return true;
  uint64_t t0 = 0;
  for (unsigned i = 1; !__all_sync(0xffffffffu, mbar_try_wait(b, parity)); ++i) {
    if ((i & 63u) == 0) {
      const uint64_t t = globaltimer_ns();
      if (t0 == 0) t0 = t;
      if (__any_sync(0xffffffffu, t - t0 > timeout_ns || i > (1u << 28))) {
        atomicCAS(err, 0, kDevErrTimeout);
        return false;
      }
    }
  }
  return true;
}

// Grid-wide sums of n values kept as per-CTA pairs part[i * G + cta], into
// out[i]; the same order in every CTA.  A warp takes eight values at once.
__device__ __forceinline__ void sum_over_ctas(const df* part, int n, int G, df* out) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i0 = 8 * w; i0 < n; i0 += 8 * (kWorkThreads / 32)) {
    df v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = df_zero();
    for (int c0 = 0; c0 < G; c0 += 32) {
      const int c = c0 + lane;
      float2 t[8];
#pragma unroll
      for (int e = 0; e < 8; ++e)
        t[e] = (c < G && i0 + e < n) ? __ldcg(reinterpret_cast<const float2*>(part + (size_t)(i0 + e) * G + c))
                                     : make_float2(0.f, 0.f);
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = df_add(v[e], df{t[e].x, t[e].y});
    }
    const df s = df_warp_sum8(v);
    if (lane < 8 && i0 + lane < n) out[i0 + lane] = s;
  }
}

// The producer warp.  Passes `first` to `last` - 1 one after another: the chunks of the CTA's units in order, dealt to the
// groups in turn (a unit is padded to whole rounds with empty chunks, so
// every group sees every unit), then a round of end marks.  The lanes take a
// block of up to S chunks, one each: a lane waits until its stage's last chunk
// has been read, puts NCX values of each of the chunk's columns (rows(pass, i),
// i < NCX; null: zeros) and the column index beside it, and issues the copy.
struct Stream {
  const void* R;
  int64_t N;
  uint32_t colbytes;
  unsigned char* ring;
  StageMeta* meta;
  float* cxs;              // [S][cx_stride], column e, row i of a chunk at e * NCX + i
  int cx_stride;
  uint64_t *full, *empty;
  int S, NG, G, cta;
  Units units;
  int nunits, dynamic;
  unsigned* work;          // unit counter of pass k at work[k - first]
  volatile int* quit;
  int* err;
  uint64_t timeout_ns;
};
template <int CW, int NCX, typename Rows>
__device__ __forceinline__ void produce(const Stream& a, int first, int last, Rows rows) {
  const int lane = threadIdx.x & 31;
  const int S = a.S, NG = a.NG;
  const int64_t N = a.N;
  const uint32_t stagebytes = (uint32_t)CW * a.colbytes;
  int* err = a.err;
  const uint64_t tmo = a.timeout_ns;
  const int BL = S < 32 ? S : 32;
  unsigned base = 0;                          // chunks issued before this block
  bool ok = true;
  float c[CW * NCX];
  auto put = [&](bool mine, int64_t j, int n, int u, int count) {   // count: lanes of the block
    const unsigned q = base + (unsigned)lane;
    const unsigned st = q % (unsigned)S, round = q / (unsigned)S;
    bool todo = mine;
    uint64_t t0 = 0;
    for (unsigned i = 1; __any_sync(0xffffffffu, todo); ++i) {
      if (todo && (round == 0 || mbar_try_wait(a.empty + st, (round - 1) & 1u))) {
        todo = false;
#pragma unroll
        for (int e = 0; e < CW * NCX; ++e) a.cxs[st * a.cx_stride + e] = c[e];
        a.meta[st].j = j;
        a.meta[st].n = n;
        a.meta[st].u = u;
        if (n > 0) {
          mbar_arrive_expect_tx(a.full + st, (uint32_t)n * a.colbytes);
          bulk_load(a.ring + (size_t)st * stagebytes,
                    reinterpret_cast<const unsigned char*>(a.R) + (size_t)j * a.colbytes, (uint32_t)n * a.colbytes,
                    a.full + st);
        } else {
          mbar_arrive(a.full + st);
        }
      }
      if ((i & 63u) == 0) {                   // bounded
        const uint64_t tn = globaltimer_ns();
        if (t0 == 0) t0 = tn;
        if (*a.quit) ok = false;
        if (tn - t0 > tmo || i > (1u << 28)) {
          if (todo) atomicCAS(err, 0, kDevErrTimeout);
          ok = false;
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
      }
    }
    if (ok) {
      base += (unsigned)count;
    } else {
      // this block's copies that were issued land before the CTA exits (bounded)
      if (mine && !todo) mbar_wait_bounded(a.full + st, round & 1u, err, tmo);
      __syncwarp();
    }
  };
  for (int k = first; k < last && ok; ++k) {
    auto grab = [&]() -> unsigned { return lane == 0 ? atomicAdd(a.work + (k - first), 1u) : 0u; };   // lane 0 has it
    // the first unit is the CTA's own (a CTA that runs ahead into this pass must
    // not take two large ones); the others come from the counter, asked for
    // a block before they are needed
    int64_t u = a.cta;
    while (u < a.nunits && ok) {
      unsigned unext = 0u;
      int64_t lo, hi;
      unit_range(a.units, N, u, lo, hi);
      const int64_t chunks = (hi - lo + CW - 1) / CW;
      const int64_t total = (chunks > 0 ? (chunks + NG - 1) / NG : 1) * NG;
      auto load_c = [&](int64_t i) {          // the rows on chunk i of the unit
        const int64_t j = lo + i * CW;
#pragma unroll
        for (int r = 0; r < NCX; ++r) {
          const float* cn = rows(k, r);
#pragma unroll
          for (int e = 0; e < CW; ++e) c[e * NCX + r] = cn && i < total && j + e < hi ? __ldcg(cn + j + e) : 0.f;
        }
      };
      load_c(lane);
      for (int64_t i0 = 0; i0 < total && ok; i0 += BL) {
        const int count = (int)(total - i0 < BL ? total - i0 : BL);
        if (a.dynamic && i0 + BL >= total) unext = grab();
        const int64_t j = lo + (i0 + lane) * CW;
        const int n = j < hi ? (int)(hi - j < CW ? hi - j : CW) : 0;
        put(lane < count, j, n, (int)u, count);
        if (i0 + BL < total) load_c(i0 + BL + lane);
      }
      u = a.dynamic ? (int64_t)a.G + (int64_t)__shfl_sync(0xffffffffu, unext, 0) : (int64_t)a.nunits;
    }
    for (int i0 = 0; i0 < NG && ok; i0 += BL) {
#pragma unroll
      for (int e = 0; e < CW * NCX; ++e) c[e] = 0.f;
      const int count = NG - i0 < BL ? NG - i0 : BL;
      put(lane < count, 0, -1, 0, count);
    }
  }
  // earlier copies still in flight land before the CTA exits (bounded)
  if (!ok && lane == 0) {
    for (unsigned d = base > (unsigned)S ? base - (unsigned)S : 0u; d < base; ++d)
      mbar_wait_bounded(a.full + d % (unsigned)S, (d / (unsigned)S) & 1u, err, tmo);
  }
}

// ------------------------------------------------------------- the kernel
template <int NR, int CW, bool BF16>
__global__ void __launch_bounds__(kDeferThreads, 1) defer_kernel(DeferArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  typedef Vec<BF16> V;
  typedef typename V::raw raw;
  constexpr int VR = V::kRows, VH = VR / 2, ELEM = BF16 ? 2 : 4;
  if (a.ctrl->stopped) return;                    // (set by an earlier launch: the same in every CTA)
  const int G = gridDim.x, cta = blockIdx.x;
  const int ld = a.ld, K = a.K, S = a.S, NG = a.NG, GS = a.GS;
  const int64_t N = a.N;
  const DeferSmem L = defer_smem(ld, K, G, S, CW, ELEM);
  unsigned char* ring = smem + L.ring;
  float* bos = reinterpret_cast<float*>(smem + L.bo);
  float* bns = reinterpret_cast<float*>(smem + L.bn);
  df* xw = reinterpret_cast<df*>(smem + L.xw);
  df* sums = reinterpret_cast<df*>(smem + L.sums);
  df* accd = reinterpret_cast<df*>(smem + L.accd);
  float* bks = reinterpret_cast<float*>(smem + L.bk);
  StageMeta* meta = reinterpret_cast<StageMeta*>(smem + L.meta);
  float* cxs = reinterpret_cast<float*>(smem + L.cx);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + L.bars);
  uint64_t* empty = full + S;
  __shared__ volatile int quit;                   // -1: a computing thread gave up waiting for a stage; 1: the CTA leaves
  int* s_ok = reinterpret_cast<int*>(smem + L.misc);
  df* cc0 = reinterpret_cast<df*>(smem + L.misc + 16);             // ||c_1||^2 of the refresh
  int* err = &a.ctrl->err;
  const uint64_t tmo = a.timeout_ns;
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const uint32_t colbytes = (uint32_t)ld * ELEM;
  const uint32_t stagebytes = (uint32_t)CW * colbytes;

  if (t < S) {
    mbar_init(full + t, 1);
    mbar_init(empty + t, GS / 32);
  }
  if (t == 0) quit = 0;
  fence_mbar_init();
  __syncthreads();

  if (w == kWorkThreads / 32) {
    // ------------------------------------------------------------ producer
    // (pass k takes c_{k+1} along)
    Stream p{a.R, N, colbytes, ring, meta, cxs, kMaxCw, full, empty, S, NG, G, cta, a.units, a.nunits, a.dynamic,
             a.work + (a.npart_first > 0 ? 1 : 0), &quit, err, tmo};
    produce<CW, 1>(p, a.npart_first > 0 ? 0 : -1, K,
                   [&](int k, int) -> const float* { return k + 1 < K ? a.C + (int64_t)(k + 1) * N : nullptr; });
    return;
  }

  // own rows (phase A) and own columns (phases B, F)
  const int rpc = defer_rows(ld, G), rst = rpc | 1;
  const int r0 = cta * rpc, nrows = max(0, min(ld, r0 + rpc) - r0);
  int64_t jlo, jhi;
  if (a.dynamic) {
    jlo = N * cta / G;
    jhi = N * (cta + 1) / G;
  } else {
    unit_range(a.units, N, cta, jlo, jhi);
  }

  if (w > kWorkThreads / 32) {
    // --------------------------------------------- side warps: phase B of each k
    const int ts = t - kWorkThreads - 32, ws = ts >> 5;
    df* xwarp = xw + (size_t)(16 + ws) * 2 * (K + 1);
    for (int k = 0; k < K; ++k) {
      side_wait(2);
      if (quit > 0) return;
      const bool more = k + 1 < K;
      const float* cn_row = a.C + (int64_t)(more ? k + 1 : 0) * N;
      for (int e = lane; e < 2 * (K + 1); e += 32) xwarp[e] = df_zero();
      __syncwarp();
      for (int64_t j0 = jlo + ts; j0 - ts < jhi; j0 += (int64_t)kTiles * kSideThreads) {
        float cn[kTiles];
        df corr[kTiles];
#pragma unroll
        for (int i = 0; i < kTiles; ++i) {
          const int64_t j = j0 + i * kSideThreads;
          cn[i] = j < jhi && more ? __ldcg(cn_row + j) : 0.f;
          corr[i] = df_zero();
        }
        for (int l0 = 0; l0 < k; l0 += 4) {
          df v[8];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int l = l0 + e < k ? l0 + e : 0;
            const bool lin = l0 + e < k;
            float cp[kTiles], co[kTiles];
#pragma unroll
            for (int i = 0; i < kTiles; ++i) {
              const int64_t j = j0 + i * kSideThreads;
              const bool in = lin && j < jhi;
              cp[i] = in ? __ldcg(a.C + (int64_t)l * N + j) : 0.f;
              co[i] = in ? __ldcg(a.Co + (int64_t)l * N + j) : 0.f;
            }
            const df yo = sums[2 * l], yn = sums[2 * l + 1];
            v[2 * e] = df_zero();
            v[2 * e + 1] = df_zero();
#pragma unroll
            for (int i = 0; i < kTiles; ++i) {
              corr[i] = df_fma(cp[i], yn, corr[i]);       // c_l' (b_k'.b_l')
              corr[i] = df_fma(-co[i], yo, corr[i]);      // c_l (b_k'.b_l)
              v[2 * e] = df_fma(co[i], cn[i], v[2 * e]);
              v[2 * e + 1] = df_fma(cp[i], cn[i], v[2 * e + 1]);
            }
          }
          if (more) {
            const df q = df_warp_sum8(v);
            if (lane < 8 && l0 + (lane >> 1) < k) xwarp[2 * l0 + lane] = df_add(xwarp[2 * l0 + lane], q);
          }
        }
#pragma unroll
        for (int i = 0; i < kTiles; ++i) {
          const int64_t j = j0 + i * kSideThreads;
          if (j < jhi) __stcg(reinterpret_cast<float2*>(a.corr + j), make_float2(corr[i].h, corr[i].l));
        }
      }
      side_arrive(3);
    }
    return;
  }

  // ------------------------------------------------------- computing warps
  unsigned nbar = 0;
  // Leaving: the side warps are let on once more and see it.  Where they may be
  // in phase B (busy), they finish it first, so that all of them see it at the same start.
#define DID_DEFER_LEAVE(busy)   \
  do {                          \
    if (busy) side_wait(3);     \
    if (t == 0) quit = 1;       \
    side_arrive(2);             \
    return;                     \
  } while (0)
#define DID_DEFER_GRID_SYNC(busy)                                                                              \
  do {                                                                                                         \
    ++nbar;                                                                                                    \
    if (!work_grid_sync(&a.ctrl->bar, nbar * (unsigned)G + (unsigned)a.bar_extra, err, tmo, s_ok, &quit))       \
      DID_DEFER_LEAVE(busy);                                                                                   \
  } while (0)

  const int g = t / GS, lt = t - g * GS;          // column group, place in it
  const int W = GS >> 5, wg = (t - g * GS) >> 5;  // warps of a group, this warp's place
  const int nvec = ld / VR;
  const bool last_ok = lt + (NR - 1) * GS < nvec;
  unsigned cst = (unsigned)g % (unsigned)S, cph = ((unsigned)g / (unsigned)S) & 1u;   // next chunk of this group
  const bool stamps = a.tstamp != nullptr && cta == 0 && t == 0;

  df* xwarp = xw + (size_t)w * 2 * (K + 1);       // this warp's sums: c_l.c at 2l, c_l'.c at 2l + 1; ||c||^2 at 2K

  // k = -1 (where the launch has no partials for c_1): phase S alone, for the
  // partials of R_s c_1^T, and ||c_1||^2 in phase F
  for (int k = a.npart_first > 0 ? 0 : -1; k < K; ++k) {
    const bool rec = stamps && k >= 0 && k < a.tstamp_cap;
    if (rec) a.tstamp[4 * k + 0] = globaltimer_ns();
    if (k >= 0) {
    // ------------------------------------------------------------ phase A
    // ||c_k||^2 and, for l < k, c_l.c_k (sums[2l]) and c_l'.c_k (sums[2l+1])
    const bool given = k == 0 && a.npart_first > 0;   // the refresh's partials
    if (given) {
      if (w == 0) {
        const double cc = warp_sum_global_f64(a.CC0, a.npart_first, 1);
        const float h = (float)cc;
        if (lane == 0) *cc0 = df{h, (float)(cc - (double)h)};
      }
    } else {
      sum_over_ctas(a.Xp, 2 * k + 1, G, sums);
    }
    // partial rows: thread (row quad, subset sub) adds rows sub, sub + SU, ... of P
    const int U = given ? a.npart_first : a.npart;
    const int nq = rpc / 4, SU = kWorkThreads / nq;
    df* acca = xw;                                 // [SU][rpc]
    const int quad = t % nq, sub = t / nq;
    if (sub < SU && 4 * quad < nrows) {            // (ld and rpc are multiples of four)
      df q[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) q[e] = df_zero();
      const float* Pr = a.P + r0 + 4 * quad;
      for (int gi0 = sub; gi0 < U; gi0 += 8 * SU) {
        float4 v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int gi = gi0 + e * SU;
          v[e] = gi < U ? __ldcg(reinterpret_cast<const float4*>(Pr + (size_t)gi * ld)) : make_float4(0.f, 0.f, 0.f, 0.f);
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
      for (int e = 0; e < 4; ++e) acca[(size_t)sub * rpc + 4 * quad + e] = q[e];
    }
    work_sync();                                   // (also publishes sums)
    // b_k' of the slice: LPR lanes per row add the subsets and the pending
    // terms sum_l b_l (c_l.c_k) - b_l' (c_l'.c_k)
    {
      const int LPR = rpc >= 32 ? 8 : 32;
      const int e0 = t & (LPR - 1);
      const df cc = given ? *cc0 : sums[2 * k];
      for (int row0 = 0; row0 < rpc; row0 += kWorkThreads / LPR) {
        const int row = row0 + t / LPR;
        const bool in = row < nrows;
        const float b_old = in ? __ldcg(a.B + (size_t)k * ld + r0 + row) : 0.f;
        df q = df_zero();
        if (in) {
          for (int e = e0; e < SU; e += LPR) q = df_add(q, acca[(size_t)e * rpc + row]);
          for (int l = e0; l < k; l += LPR) {
            q = df_fma(bos[l * rst + row], sums[2 * l], q);
            q = df_fma(-bns[l * rst + row], sums[2 * l + 1], q);
          }
        }
        for (int m = LPR / 2; m >= 1; m >>= 1) q = df_add(q, df_shfl_xor(q, m));
        if (in && e0 == 0) {
          float b_new = b_old;
          if (cc.h > 0.f) {
            const df v = df_add(df{b_old, 0.f}, df_div(q, cc));
            b_new = v.h > 0.f ? v.h : 0.f;
          }
          bos[k * rst + row] = b_old;
          bns[k * rst + row] = b_new;
          bks[row] = b_new;
          __stcg(a.Bo + (size_t)k * ld + r0 + row, b_old);
          __stcg(a.B + (size_t)k * ld + r0 + row, b_new);
          if (!(cc.h > 0.f) && cta == 0 && row == 0) atomicAdd(a.degen, 1ull);
        }
      }
      work_sync();
    }
    // the slice's sums b_k'.b_l, b_k'.b_l' (l < k) and b_k'.b_k, b_k'.b_k' (l = k):
    // thread (l, part of the rows)
    {
      int LP = 32;
      while (LP < k + 1) LP *= 2;
      const int parts = kWorkThreads / LP;
      const int l = t & (LP - 1), part = t / LP;
      df yo = df_zero(), yn = df_zero();
      if (l <= k) {
        for (int r = part; r < nrows; r += parts) {
          const float b = bks[r];
          yo = df_fma(b, bos[l * rst + r], yo);
          yn = df_fma(b, bns[l * rst + r], yn);
        }
      }
      accd[t] = yo;
      accd[kWorkThreads + t] = yn;
      work_sync();
      if (t <= k) {
        df so = accd[t], sn = accd[kWorkThreads + t];
        for (int e = 1; e < parts; ++e) {
          so = df_add(so, accd[e * LP + t]);
          sn = df_add(sn, accd[kWorkThreads + e * LP + t]);
        }
        __stcg(reinterpret_cast<float2*>(a.Yp + (size_t)(2 * t) * G + cta), make_float2(so.h, so.l));
        __stcg(reinterpret_cast<float2*>(a.Yp + (size_t)(2 * t + 1) * G + cta), make_float2(sn.h, sn.l));
      }
    }
    DID_DEFER_GRID_SYNC(false);
    if (rec) a.tstamp[4 * k + 1] = globaltimer_ns();

    sum_over_ctas(a.Yp, 2 * k + 2, G, sums);
    work_sync();
    if (!(sums[2 * k + 1].h > 0.f) && cta == 0 && t == 0) atomicAdd(a.degen, 1ull);
    if (lane < 3) xwarp[lane < 2 ? 2 * k + lane : 2 * K] = df_zero();
    side_arrive(2);                              // the side warps begin phase B
    } else if (lane == 0) {
      xwarp[2 * K] = df_zero();
    }
    // b_k' of this thread's rows
    float2 bn[NR][VH];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int q = lt + r * GS;
      const bool in = r < NR - 1 || last_ok;
#pragma unroll
      for (int e = 0; e < VR; e += 4) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in && k >= 0) v = __ldcg(reinterpret_cast<const float4*>(a.B + (size_t)k * ld + (size_t)q * VR + e));
        bn[r][e / 2] = make_float2(v.x, v.y);
        bn[r][e / 2 + 1] = make_float2(v.z, v.w);
      }
    }
    const bool more = k + 1 < K;                 // the next step needs the sums with c_{k+1}
    const float* cn_row = a.C + (int64_t)(more ? k + 1 : 0) * N;

    // ------------------------------------------------------------ phase S
    {
      // The partials of a unit in two levels (float32 residual): 16 chunks are
      // summed in p and added to pt, which keeps the chains of additions short (a unit holds
      // up to about 800 columns; one chain for it lost a bit of b).
      constexpr bool kTwo = !BF16 && NR <= 6;
      float2 p[NR][VH], pt[kTwo ? NR : 1][VH];
#pragma unroll
      for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int h = 0; h < VH; ++h) p[r][h] = pt[kTwo ? r : 0][h] = make_float2(0.f, 0.f);
      int cu = -1, np = 0;
      auto collect = [&]() {
        if (kTwo) {
#pragma unroll
          for (int r = 0; r < NR; ++r)
#pragma unroll
            for (int h = 0; h < VH; ++h) {
              float2& q = pt[kTwo ? r : 0][h];
              q = make_float2(q.x + p[r][h].x, q.y + p[r][h].y);
              p[r][h] = make_float2(0.f, 0.f);
            }
          np = 0;
        }
      };
      auto flush = [&](int u) {
        if (!more) return;
        if (kTwo) {
          collect();
#pragma unroll
          for (int r = 0; r < NR; ++r)
#pragma unroll
            for (int h = 0; h < VH; ++h) {
              p[r][h] = pt[kTwo ? r : 0][h];
              pt[kTwo ? r : 0][h] = make_float2(0.f, 0.f);
            }
        }
        float* Pu = a.P + (size_t)(u * NG + g) * ld;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const int q = lt + r * GS;
          if (r < NR - 1 || last_ok) {
#pragma unroll
            for (int e = 0; e < VR; e += 4)
              __stcg(reinterpret_cast<float4*>(Pu + (size_t)q * VR + e),
                     make_float4(p[r][e / 2].x, p[r][e / 2].y, p[r][e / 2 + 1].x, p[r][e / 2 + 1].y));
          }
#pragma unroll
          for (int h = 0; h < VH; ++h) p[r][h] = make_float2(0.f, 0.f);
        }
      };
      while (true) {
        if (!stage_wait(full + cst, cph, err, tmo)) {
          quit = -1;                               // the CTA leaves after this phase
          break;
        }
        const int64_t j = meta[cst].j;
        const int n = meta[cst].n, u = meta[cst].u;
        const unsigned st = cst;
        cst += (unsigned)NG;
        while (cst >= (unsigned)S) {
          cst -= (unsigned)S;
          cph ^= 1u;
        }
        if (n < 0) {                               // the pass is over: give the mark's stage back
          __syncwarp();
          if (lane == 0) mbar_arrive(empty + st);
          break;
        }
        if (u != cu) {
          if (cu >= 0) flush(cu);
          cu = u;
        } else if (kTwo && ++np == 16) {
          collect();
        }
        const raw* col = reinterpret_cast<const raw*>(ring + (size_t)st * stagebytes) + lt;
        float2 d[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) d[c] = make_float2(0.f, 0.f);
        if (n == CW) {
          float cx[CW];
#pragma unroll
          for (int c = 0; c < CW; ++c) cx[c] = cxs[st * kMaxCw + c];
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            if (r < NR - 1 || last_ok) {
              raw x[CW];
#pragma unroll
              for (int c = 0; c < CW; ++c) x[c] = col[(size_t)c * nvec + r * GS];
#pragma unroll
              for (int c = 0; c < CW; ++c) {
                float f[VR];
                V::unpack(x[c], f);
                const float2 c2 = make_float2(cx[c], cx[c]);
#pragma unroll
                for (int h = 0; h < VH; ++h) {
                  const float2 f2 = make_float2(f[2 * h], f[2 * h + 1]);
                  d[c] = __ffma2_rn(bn[r][h], f2, d[c]);
                  p[r][h] = __ffma2_rn(f2, c2, p[r][h]);
                }
              }
            }
          }
        } else {
          // the unit's last chunk (or none): only the columns that are there
#pragma unroll
          for (int c = 0; c < CW; ++c) {
            if (c < n) {
              const float cx = cxs[st * kMaxCw + c];
              const float2 c2 = make_float2(cx, cx);
#pragma unroll
              for (int r = 0; r < NR; ++r) {
                if (r < NR - 1 || last_ok) {
                  float f[VR];
                  V::unpack(col[(size_t)c * nvec + r * GS], f);
#pragma unroll
                  for (int h = 0; h < VH; ++h) {
                    const float2 f2 = make_float2(f[2 * h], f[2 * h + 1]);
                    d[c] = __ffma2_rn(bn[r][h], f2, d[c]);
                    p[r][h] = __ffma2_rn(f2, c2, p[r][h]);
                  }
                }
              }
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + st);
        // this warp's part of the CW dot products: lanes 0, 32/CW, ... get one each
        float v[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) v[c] = d[c].x + d[c].y;
        int m = 16;
#pragma unroll
        for (int h = CW / 2; h >= 1; h >>= 1) {
          const bool up = (lane & m) != 0;
#pragma unroll
          for (int i = 0; i < h; ++i) {
            const float send = up ? v[i] : v[i + h];
            const float keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, m);
          }
          m >>= 1;
        }
#pragma unroll
        for (int mm = 16 / CW; mm >= 1; mm >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], mm);
        const int c = lane / (32 / CW);
        if ((lane & (32 / CW - 1)) == 0 && c < n) __stcg(a.T + (size_t)(j + c) * W + wg, v[0]);
      }
      if (cu >= 0) flush(cu);
    }
    if (rec) a.tstamp[4 * k + 2] = globaltimer_ns();
    if (a.dynamic) {
      DID_DEFER_GRID_SYNC(k >= 0);
    } else {
      __threadfence_block();
      work_sync();
      if (quit) DID_DEFER_LEAVE(k >= 0);
    }

    // ------------------------------------------------------------ phase F
    if (k < 0) {
      df cc = df_zero();
      for (int64_t j = jlo + t; j < jhi; j += kWorkThreads) {
        const float c = __ldcg(cn_row + j);
        cc = df_fma(c, c, cc);
      }
      df v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = e == 0 ? cc : df_zero();
      cc = df_warp_sum8(v);
      if (lane == 0) xwarp[2 * K] = cc;
    } else {
    side_wait(3);
    const df bob = sums[2 * k], bb = sums[2 * k + 1];
    const bool cdeg = !(bb.h > 0.f);
    const df inv_bb = cdeg ? df_zero() : df_div(df{1.f, 0.f}, bb);
    for (int64_t j0 = jlo; j0 < jhi; j0 += (int64_t)kTiles * kWorkThreads) {
      float c_old[kTiles], cn[kTiles];
      df q[kTiles];
#pragma unroll
      for (int i = 0; i < kTiles; ++i) {
        const int64_t j = j0 + t + i * kWorkThreads;
        const bool in = j < jhi;
        c_old[i] = in ? __ldcg(a.C + (int64_t)k * N + j) : 0.f;
        cn[i] = in && more ? __ldcg(cn_row + j) : 0.f;
        // b_k'^T R_s - the pending terms
        const float2 cr = in ? __ldcg(reinterpret_cast<const float2*>(a.corr + j)) : make_float2(0.f, 0.f);
        q[i] = df{-cr.x, -cr.y};
        if (in) {
          const float* Tj = a.T + (size_t)j * W;
          if (W >= 4) {
            for (int e = 0; e < W; e += 4) {
              const float4 x = __ldcg(reinterpret_cast<const float4*>(Tj + e));
              df_acc(q[i], x.x);
              df_acc(q[i], x.y);
              df_acc(q[i], x.z);
              df_acc(q[i], x.w);
            }
          } else {
            for (int e = 0; e < W; ++e) df_acc(q[i], __ldcg(Tj + e));
          }
        }
      }
      df v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = df_zero();
#pragma unroll
      for (int i = 0; i < kTiles; ++i) {
        const int64_t j = j0 + t + i * kWorkThreads;
        if (j < jhi) {
          // (b_k'^T R + (b_k'.b_k) c_k) / ||b_k'||^2
          float c_new = c_old[i];
          if (!cdeg) {
            const float tt = df_mul_f32(df_fma(c_old[i], bob, q[i]), inv_bb);
            c_new = tt > 0.f ? tt : 0.f;
          }
          __stcg(a.C + (int64_t)k * N + j, c_new);
          __stcg(a.Co + (int64_t)k * N + j, c_old[i]);
          v[0] = df_fma(c_old[i], cn[i], v[0]);
          v[1] = df_fma(c_new, cn[i], v[1]);
          v[2] = df_fma(cn[i], cn[i], v[2]);
        }
      }
      if (more) {
        const df s8 = df_warp_sum8(v);
        if (lane < 3) {
          df* x = xwarp + (lane < 2 ? 2 * k + lane : 2 * K);
          *x = df_add(*x, s8);
        }
      }
    }
    }
    if (!more) break;
    work_sync();
    // the CTA's sums, warps in order: entries 0 .. 2k - 1 of the side warps,
    // then those of l = k and ||c_{k+1}||^2 of the computing warps
    for (int i = t; i < 2 * k + 3; i += kWorkThreads) {
      const int src = i < 2 * k + 2 ? i : 2 * K;
      const int e0 = i < 2 * k ? 16 : 0, e1 = i < 2 * k ? 20 : 16;
      df s = df_zero();
      for (int e = e0; e < e1; ++e) s = df_add(s, xw[(size_t)e * 2 * (K + 1) + src]);
      __stcg(reinterpret_cast<float2*>(a.Xp + (size_t)i * G + cta), make_float2(s.h, s.l));
    }
    DID_DEFER_GRID_SYNC(false);
    if (rec) a.tstamp[4 * k + 3] = globaltimer_ns();
  }
#undef DID_DEFER_GRID_SYNC
#undef DID_DEFER_LEAVE
  if (stamps && K - 1 < a.tstamp_cap) a.tstamp[4 * (K - 1) + 3] = globaltimer_ns();
}

const void* defer_func_f32(int NR, int CW);
const void* defer_func_bf16(int NR, int CW);

}  // namespace defer_impl
}  // namespace did
