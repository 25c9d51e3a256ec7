// Sweeps of a residual that fits the SMs' shared memory: R stays there for the
// whole launch, and the CTAs exchange flagged words instead of meeting at
// grid barriers.
//
// Each CTA owns a range of columns of R and C and, for the b updates, a slice
// of rows.  Per k of the interleaved order (Section 2, HALS closed forms):
//   1  every CTA has the partials of R c_k^T over its columns (formed while the
//      previous step updated R) and sends them, with ||c_k||^2 over its columns, as
//      words (value, step number);
//   2  the owner of a row adds the CTAs' words in order, forms b_k'
//      (sol:b_i) and sends (b_k', step, b_k, step);
//   3  every CTA takes all rows of b_k' and b_k, forms ||b_k'||^2 and
//      b_k'.b_k, updates c_k on its columns (up:c) and R in shared memory, and
//      forms the partials for k + 1 in the same loop.
// The C-first order (Algorithm 2) runs its C step without any exchange (b is
// fixed and the columns are local), its B step by the same two exchanges, and
// one grid barrier per sweep, after which the new B is read back.
//
// What bounds it: latency, two one-way trips through L2 per k.  A word
// carries its step number in the same 8 bytes, so the receiver polls the data
// itself: no fence, no atomic, and no load after the barrier.  The sweep kernel's
// per-k cost on these sizes is 27 to 32 us (two grid barriers with the
// loads behind them); here 6.5 us at 200 x 1000 (32 CTAs), 8.6 us at 1024 x
// 2414 (76 CTAs), of which the exchange takes 2.4 and 3.7.  A word is
// overwritten only after its readers have used it: a CTA sends the partials of step s + 1
// after it has all of b'(s), and b'(s) is sent after the owner has read every
// CTA's partials of step s.
//
// Every wait is bounded; on expiry the error word is set and all CTAs leave.
#include "did_internal.cuh"
#include "did_pair.cuh"

#include <algorithm>
#include <type_traits>

namespace did {

namespace {

constexpr int kResThreads = 512;
constexpr int kResWarps = kResThreads / 32;

struct ResArgs {
  void* R;             // ld x N residual in global memory (float or bfloat16), read at the start, written at the end
  float* B;            // ld x K
  float* C;            // K x N
  uint2* Pw;           // [grid][ld + 8] words: partial rows, then ||c||^2 (hi, lo) of even and of odd steps,
                       // ||R||^2 (hi, lo) of even and of odd sweeps
  uint4* Bw;           // [ld] words (b', step, b, step)
  Ctrl* ctrl;
  double* trace;
  unsigned long long* degen;
  int64_t N;
  int ld, K;
  int nc;              // columns of a CTA
  int bf16;
  int n_sweeps, order;
  unsigned step0;      // step numbers of this launch begin after step0
  int stop_rule;
  double tol, f_prev, f0;
  int bar_extra;       // test hook: > 0 makes the first wait one for a word that never comes
  uint64_t timeout_ns;
  uint64_t* tstamp;
  int tstamp_cap;
  int cta_begin, cta_count;   // several instances in one launch: the CTAs of this one
};

struct ResSmem {
  size_t R, bn, bo, C, cn, vals, ps, red, brow, misc, total;   // (K only for the own rows of B)
};
__host__ __device__ __forceinline__ ResSmem res_smem(int ld, int K, int nc, int grid) {
  ResSmem L;
  const int rpc = (ld + grid - 1) / grid;
  size_t o = 0;
  L.R = o;    o += (size_t)nc * ld * 4;
  L.bn = o;   o += (size_t)ld * 4;
  L.bo = o;   o += (size_t)ld * 4;
  const size_t ncp = ((size_t)nc + 3) & ~(size_t)3;                  // rows of C padded for 16-byte loads
  L.C = o;    o += (size_t)2 * ncp * 4;                              // rows k and k + 1 of C on the own columns
  L.cn = o;   o += (size_t)2 * ncp * 4;                              // c_k before and after its update
  L.vals = o; o += ((size_t)(rpc + 4) * grid * 4 + 15) & ~(size_t)15;
  L.ps = o;   o += (size_t)kResThreads * 4;                          // a short column's partials by parts of the columns
  L.brow = o; o += ((size_t)rpc * K * 4 + 15) & ~(size_t)15;         // own rows of B
  L.red = o;  o += (size_t)kResWarps * 4 * 8;
  L.misc = o; o += 64;
  L.total = o;
  return L;
}

__device__ __forceinline__ void st_word(uint2* p, float v, unsigned step) {
  const unsigned long long x = (unsigned long long)__float_as_uint(v) | ((unsigned long long)step << 32);
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(x) : "memory");
}
__device__ __forceinline__ uint2 ld_word(const uint2* p) {
  unsigned long long x;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(x) : "l"(p) : "memory");
  return make_uint2((unsigned)x, (unsigned)(x >> 32));
}

// Two words (each valid by its own step number).
__device__ __forceinline__ uint4 ld_words(const uint4* p) {
  unsigned long long x, y;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
  return make_uint4((unsigned)x, (unsigned)(x >> 32), (unsigned)y, (unsigned)(y >> 32));
}

// Poll limit: looked at every 64 polls.
struct Poll {
  uint64_t t0 = 0;
  unsigned i = 0;
  __device__ __forceinline__ bool expired(int* err, uint64_t timeout_ns) {
    if ((++i & 63u) != 0) return false;
    const uint64_t t = globaltimer_ns();
    if (t0 == 0) t0 = t;
    if (ld_volatile(err) != 0) return true;
    if (t - t0 > timeout_ns || i > (1u << 28)) {
      atomicCAS(err, 0, kDevErrTimeout);
      return true;
    }
    return false;
  }
};

__device__ __forceinline__ void resident_body(const ResArgs& a, const int cta, const int G) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const int ld = a.ld, K = a.K;
  const int64_t N = a.N;
  const ResSmem L = res_smem(ld, K, a.nc, G);
  const int ncp = (a.nc + 3) & ~3;
  float* R = reinterpret_cast<float*>(smem + L.R);
  float* bn = reinterpret_cast<float*>(smem + L.bn);
  float* bo = reinterpret_cast<float*>(smem + L.bo);
  float* Cs = reinterpret_cast<float*>(smem + L.C);
  float* cold = reinterpret_cast<float*>(smem + L.cn);
  float* cnew = cold + ncp;
  float* vals = reinterpret_cast<float*>(smem + L.vals);
  float* ps = reinterpret_cast<float*>(smem + L.ps);
  float* brow = reinterpret_cast<float*>(smem + L.brow);
  df* red = reinterpret_cast<df*>(smem + L.red);
  volatile int* bad = reinterpret_cast<volatile int*>(smem + L.misc);
  int* err = &a.ctrl->err;
  const uint64_t tmo = a.timeout_ns;
  const int64_t j0 = (int64_t)cta * a.nc;
  const int nc = (int)(j0 < N ? (N - j0 < a.nc ? N - j0 : a.nc) : 0);
  const int rpc = (ld + G - 1) / G;
  const int r0 = cta * rpc, nrows = max(0, min(ld, r0 + rpc) - r0);
  const int pw = ld + 8;                       // words of a CTA's row in Pw
  uint2* mine = a.Pw + (size_t)cta * pw;

  // own columns of R, own rows of B
  // expired waits of an exchange's first and second half and of the
  // objective: a word each, written before and read after a CTA barrier
  if (t < 3) bad[t] = 0;
  if (a.bf16) {
    const __nv_bfloat16* src = reinterpret_cast<const __nv_bfloat16*>(a.R) + (size_t)j0 * ld;
    for (int i = t; i < nc * ld; i += kResThreads) R[i] = __bfloat162float(src[i]);
  } else {
    const float4* src = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(a.R) + (size_t)j0 * ld);
    for (int i = t; i < nc * ld / 4; i += kResThreads) reinterpret_cast<float4*>(R)[i] = __ldcg(src + i);
  }
  for (int i = t; i < K * nrows; i += kResThreads) {
    const int k = i / nrows, r = i - k * nrows;
    brow[k * rpc + r] = __ldcg(a.B + (size_t)k * ld + r0 + r);
  }
  __syncthreads();

  unsigned step = a.step0;
  unsigned nbar = 0;
  double f_prev = a.f_prev;
  bool dead = false;
  const bool stamps = a.tstamp != nullptr && cta == 0 && t == 0;

  // C stays in global memory (the own columns are this CTA's alone); row k is
  // kept in shared memory for its step and the one before.
  auto crow = [&](int k) -> float* { return Cs + (k & 1) * ncp; };
  auto load_row = [&](int k) {
    for (int c = t; c < nc; c += kResThreads) crow(k)[c] = __ldcg(a.C + (size_t)k * N + j0 + c);
  };
  // ||c||^2 of a row on the own columns, sent for step `s` (one warp).
  auto send_cc = [&](const float* row, unsigned s) {
    df cc = df{0.f, 0.f};
    for (int c = lane; c < nc; c += 32) cc = df_fma(row[c], row[c], cc);
    cc = df_warp_sum(cc);
    if (lane == 0) {
      st_word(mine + ld + 2 * (s & 1), cc.h, s);
      st_word(mine + ld + 1 + 2 * (s & 1), cc.l, s);
    }
  };
  // Sum of the CTAs' words `at` and `at + 1` (a pair each) of step s, by one
  // warp; false if the wait ran out.
  auto take_pair = [&](int at, unsigned s, df& out) -> bool {
    df q = df{0.f, 0.f};
    bool ok = true;
    for (int g = lane; g < G; g += 32) {
      uint2 x, y;
      Poll poll;
      while (true) {
        x = ld_word(a.Pw + (size_t)g * pw + at);
        y = ld_word(a.Pw + (size_t)g * pw + at + 1);
        if (x.y == s && y.y == s) break;
        if (poll.expired(err, tmo)) { ok = false; break; }
      }
      if (!ok) break;
      q = df_add(q, df{__uint_as_float(x.x), __uint_as_float(y.x)});
    }
    ok = __all_sync(0xffffffffu, ok);
    out = df_warp_sum(q);
    return ok;
  };
  // Block sums of two pairs, in every thread (two barriers apart from the next use).
  auto block_pairs = [&](df& x, df& y) {
    // even lanes sum x, odd lanes y: one chain of additions instead of two
    const df send = (lane & 1) ? x : y, keep = (lane & 1) ? y : x;
    df v = df_add(keep, df_shfl_xor(send, 1));
#pragma unroll
    for (int m = 2; m <= 16; m <<= 1) v = df_add(v, df_shfl_xor(v, m));
    if (lane < 2) red[2 * w + lane] = v;
    __syncthreads();
    v = red[lane];                                 // warp lane / 2, x or y
#pragma unroll
    for (int m = 2; m <= 16; m <<= 1) v = df_add(v, df_shfl_xor(v, m));
    x = df{__shfl_sync(0xffffffffu, v.h, 0), __shfl_sync(0xffffffffu, v.l, 0)};
    y = df{__shfl_sync(0xffffffffu, v.h, 1), __shfl_sync(0xffffffffu, v.l, 1)};
  };
  // Partials of R c_1^T over the own columns, sent as step s (first step of a
  // launch or of a B step; later ones come with the update).
  auto send_first = [&](unsigned s) {
    load_row(0);
    __syncthreads();
    const float* c1 = crow(0);
    for (int r = t; r < ld; r += kResThreads) {
      float p = 0.f;
      for (int c = 0; c < nc; ++c) p = fmaf(R[c * ld + r], c1[c], p);
      st_word(mine + r, p, s);
    }
    if (w == kResWarps - 1) send_cc(c1, s);
  };
  // words of this thread in the owner's part of an exchange (the first kOwn of them)
  constexpr int kOwn = 4;
  const int per = nrows, total = nrows * G;
  int own[kOwn];
#pragma unroll
  for (int u = 0; u < kOwn; ++u) {
    const int e = t + u * kResThreads;
    own[u] = e < total ? (e / per) * pw + r0 + e % per : 0;
  }
  // b_k of step s: the owner's rows from the CTAs' words, then all rows into bn, bo.
  auto exchange = [&](int k, unsigned s) -> bool {
    // the owner's part: words (src, row) in turn, four in flight a thread
    bool ok = true;
    for (int e0 = t; e0 < total; e0 += kOwn * kResThreads) {
      const uint2* at[kOwn];
      uint2 x[kOwn];
      unsigned need = 0;
#pragma unroll
      for (int u = 0; u < kOwn; ++u) {
        const int e = e0 + u * kResThreads;
        at[u] = a.Pw;
        if (e < total) {
          if (e0 == t) {
            at[u] += own[u];
          } else {
            const int src = e / per;
            at[u] += (size_t)src * pw + r0 + (e - src * per);
          }
          need |= 1u << u;
        }
      }
      Poll poll;
      while (true) {
#pragma unroll
        for (int u = 0; u < kOwn; ++u)
          if (need & (1u << u)) x[u] = ld_word(at[u]);
#pragma unroll
        for (int u = 0; u < kOwn; ++u)
          if ((need & (1u << u)) && x[u].y == s) {
            need &= ~(1u << u);
            vals[e0 + u * kResThreads] = __uint_as_float(x[u].x);
          }
        if (!need) break;
        if (poll.expired(err, tmo)) { ok = false; break; }
      }
      if (!ok) break;
    }
    df cc = df{0.f, 0.f};
    if (w == kResWarps - 1 && nrows > 0) {
      if (!take_pair(ld + 2 * (int)(s & 1), s, cc)) ok = false;
      if (lane == 0) red[2 * kResWarps] = cc;
    }
    if (!ok) bad[0] = 1;
    __syncthreads();
    if (bad[0]) return false;
    cc = red[2 * kResWarps];
    const bool live = cc.h > 0.f;
    for (int r = w; r < nrows; r += kResWarps) {
      df q = df{0.f, 0.f};
      for (int g = lane; g < G; g += 32) q = df_add(q, df{vals[g * per + r], 0.f});
      q = df_warp_sum(q);
      if (lane == 0) {
        const float b_old = brow[k * rpc + r];
        float b_new = b_old;
        if (live) {
          const df v = df_add(df{b_old, 0.f}, df_div(q, cc));
          b_new = v.h > 0.f ? v.h : 0.f;
        }
        brow[k * rpc + r] = b_new;
        uint2* o = reinterpret_cast<uint2*>(a.Bw + r0 + r);
        st_word(o, b_new, s);
        st_word(o + 1, b_old, s);
        if (!live && r0 + r == 0) atomicAdd(a.degen, 1ull);
      }
    }
    // all rows, two in flight a thread
    for (int ra = t; ra < ld; ra += 2 * kResThreads) {
      const int rb = ra + kResThreads;
      bool na = true, nb = rb < ld;
      Poll poll;
      while (true) {
        uint4 x, y;
        if (na) x = ld_words(a.Bw + ra);
        if (nb) y = ld_words(a.Bw + rb);
        if (na && x.y == s && x.w == s) {
          bn[ra] = __uint_as_float(x.x);
          bo[ra] = __uint_as_float(x.z);
          na = false;
        }
        if (nb && y.y == s && y.w == s) {
          bn[rb] = __uint_as_float(y.x);
          bo[rb] = __uint_as_float(y.z);
          nb = false;
        }
        if (!na && !nb) break;
        if (poll.expired(err, tmo)) { ok = false; break; }
      }
      if (!ok) break;
    }
    if (!ok) bad[1] = 1;
    return true;                 // the caller's next barrier publishes bn, bo and bad
  };
  // R += bo c_old - bn c_new on the own columns (cold, cnew) and, in the same
  // loop, the partials for the row cx of C (sent as step s) and, with obj, ||R||^2.
  // (obj, a compile-time constant, keeps the sum of squares out of the other steps' loop)
  auto update_as = [&](auto objective, const float* cx, unsigned s, bool send, df& r2) {
    constexpr bool obj = decltype(objective)::value;
    // a thread per row; where the rows leave threads over, several parts of
    // the columns (up to 512 / ld, at least 8 columns each) a row
    const int parts = min(kResThreads / ld, nc / 8);
    const int chunk = parts > 1 ? ((nc + parts - 1) / parts + 3) & ~3 : nc;
    const int part = parts > 1 ? t / ld : 0;
    const int clo = min(nc, part * chunk), chi = min(nc, clo + chunk);
    for (int r = parts > 1 ? t - part * ld : t; r < ld; r += kResThreads) {
      const float x = bo[r], y = -bn[r];
      float* Rr = R + (size_t)clo * ld + r;
      float p = 0.f;
      df q = df{0.f, 0.f};                         // squares, four at a time
      int c = clo;
      for (; c + 4 <= chi; c += 4) {
        const float4 c0 = *reinterpret_cast<const float4*>(cold + c), c1 = *reinterpret_cast<const float4*>(cnew + c);
        const float4 c2 = *reinterpret_cast<const float4*>(cx + c);
        float v0 = Rr[0], v1 = Rr[ld], v2 = Rr[2 * ld], v3 = Rr[3 * ld];
        v0 = fmaf(x, c0.x, fmaf(y, c1.x, v0));
        v1 = fmaf(x, c0.y, fmaf(y, c1.y, v1));
        v2 = fmaf(x, c0.z, fmaf(y, c1.z, v2));
        v3 = fmaf(x, c0.w, fmaf(y, c1.w, v3));
        Rr[0] = v0;
        Rr[ld] = v1;
        Rr[2 * ld] = v2;
        Rr[3 * ld] = v3;
        Rr += 4 * (size_t)ld;
        p = fmaf(v0, c2.x, p);
        p = fmaf(v1, c2.y, p);
        p = fmaf(v2, c2.z, p);
        p = fmaf(v3, c2.w, p);
        if (obj) df_acc(q, fmaf(v0, v0, fmaf(v1, v1, fmaf(v2, v2, v3 * v3))));
      }
      for (; c < chi; ++c, Rr += ld) {
        const float v = fmaf(x, cold[c], fmaf(y, cnew[c], *Rr));
        *Rr = v;
        p = fmaf(v, cx[c], p);
        if (obj) df_acc(q, v * v);
      }
      if (parts > 1) {
        if (part < parts) ps[t] = p;               // ps[part * ld + r]
      } else if (send) {
        st_word(mine + r, p, s);
      }
      if (obj) r2 = df_add(r2, q);
    }
    if (parts > 1 && send) {
      __syncthreads();
      if (t < ld) {
        float p = ps[t];
        for (int e = 1; e < parts; ++e) p += ps[e * ld + t];
        st_word(mine + t, p, s);
      }
    }
  };
  auto update = [&](const float* cx, unsigned s, bool send, bool obj, df& r2) {
    if (obj)
      update_as(std::true_type{}, cx, s, send, r2);
    else
      update_as(std::false_type{}, cx, s, send, r2);
  };
  // c_k on the own columns from bn: a warp takes a column, or two where there
  // are more than warps.
  auto columns = [&](int k, const float* ck, df bb, df bob) {
    const bool cdeg = !(bb.h > 0.f);
    const float inv_bb = cdeg ? 0.f : df_div(df{1.f, 0.f}, bb).h;
    const float alpha = cdeg ? 0.f : df_div(bob, bb).h;
    if (cdeg && cta == 0 && t == 0) atomicAdd(a.degen, 1ull);
    const float4* b4 = reinterpret_cast<const float4*>(bn);
    auto finish = [&](int c, float dot) {
      const float co = ck[c];
      float cv = co;
      if (!cdeg) {
        const float v = fmaf(alpha, co, dot * inv_bb);
        cv = v > 0.f ? v : 0.f;
      }
      cold[c] = co;
      cnew[c] = cv;
      __stcg(a.C + (size_t)k * N + j0 + c, cv);
    };
    const int n4 = ld / 4;
    int c = w;
    for (; c + kResWarps < nc; c += 2 * kResWarps) {
      const float4* r4 = reinterpret_cast<const float4*>(R + (size_t)c * ld);
      const float4* q4 = reinterpret_cast<const float4*>(R + (size_t)(c + kResWarps) * ld);
      float2 d0 = make_float2(0.f, 0.f), d1 = d0, e0 = d0, e1 = d0;
      for (int i = lane; i < n4; i += 32) {
        const float4 x = r4[i], z = q4[i], y = b4[i];
        const float2 lo = make_float2(y.x, y.y), hi = make_float2(y.z, y.w);
        d0 = __ffma2_rn(make_float2(x.x, x.y), lo, d0);
        d1 = __ffma2_rn(make_float2(x.z, x.w), hi, d1);
        e0 = __ffma2_rn(make_float2(z.x, z.y), lo, e0);
        e1 = __ffma2_rn(make_float2(z.z, z.w), hi, e1);
      }
      // the lower half warp reduces the first column, the upper the second
      const float u = (d0.x + d0.y) + (d1.x + d1.y), v = (e0.x + e0.y) + (e1.x + e1.y);
      float dot = (lane < 16 ? u : v) + __shfl_xor_sync(0xffffffffu, lane < 16 ? v : u, 16);
#pragma unroll
      for (int m = 8; m >= 1; m >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, m);
      if ((lane & 15) == 0) finish(lane == 0 ? c : c + kResWarps, dot);
    }
    if (c < nc) {
      const float4* r4 = reinterpret_cast<const float4*>(R + (size_t)c * ld);
      float2 d0 = make_float2(0.f, 0.f), d1 = d0;
      for (int i = lane; i < n4; i += 32) {
        const float4 x = r4[i], y = b4[i];
        d0 = __ffma2_rn(make_float2(x.x, x.y), make_float2(y.x, y.y), d0);
        d1 = __ffma2_rn(make_float2(x.z, x.w), make_float2(y.z, y.w), d1);
      }
      const float dot = warp_sum_f32((d0.x + d0.y) + (d1.x + d1.y));
      if (lane == 0) finish(c, dot);
    }
  };

  if (a.bar_extra > 0) {         // test hook: a word nobody sends
    if (t == 0) {
      Poll poll;
      while (!poll.expired(err, tmo)) {
      }
    }
    __syncthreads();
    dead = true;
  }

  const bool inter = a.order != DID_ORDER_DID;
  if (!dead && inter) send_first(step + 1);
  for (int s = 0; s < a.n_sweeps && !dead; ++s) {
    df r2 = df{0.f, 0.f};
    if (!inter) {
      // C step: b fixed, columns local.  B is current in global memory (the
      // launch's start, or the grid barrier after the last B step).
      for (int k = 0; k < K; ++k) {
        df bb = df{0.f, 0.f}, dummy = bb;
        __syncthreads();                           // bn, bo, cold, cnew are free
        for (int r = t; r < ld; r += kResThreads) {
          const float v = __ldcg(a.B + (size_t)k * ld + r);
          bn[r] = bo[r] = v;
          bb = df_fma(v, v, bb);
        }
        load_row(k);
        block_pairs(bb, dummy);
        columns(k, crow(k), bb, bb);
        __syncthreads();
        update(cnew, 0, false, false, r2);
      }
      __syncthreads();
      send_first(step + 1);
    }
    for (int k = 0; k < K; ++k) {
      const int at = s * K + k;
      const bool rec = stamps && at < a.tstamp_cap;
      if (rec) a.tstamp[4 * at + 0] = globaltimer_ns();
      ++step;
      const int knext = k + 1 < K ? k + 1 : 0;
      const bool last = k == K - 1;
      // the next step's partials go out with this update (the last step of a
      // launch, and of a B step, sends none); its row of C is read and its
      // ||c||^2 sent before this step's exchange.  With K = 1 that row is the
      // one this step updates.  For odd K > 1 rows K - 1 and 0 fall into the
      // same buffer, so the last step takes its own row from a copy.
      const bool send = last ? inter && s + 1 < a.n_sweeps : true;
      const float* ck = crow(k);
      const float* cx = crow(knext);
      if (send && K > 1) {
        if (ck == cx) {
          __syncthreads();                         // the previous update has read cold
          for (int c = t; c < nc; c += kResThreads) cold[c] = ck[c];
          ck = cold;
          __syncthreads();
        }
        load_row(knext);
        __syncthreads();
        if (w == kResWarps - 1) send_cc(cx, step + 1);
      }
      if (!exchange(k, step)) { dead = true; break; }
      if (rec) a.tstamp[4 * at + 1] = globaltimer_ns();
      if (inter) {
        // (a thread reads only the rows it stored, so this needs no barrier)
        df bb = df{0.f, 0.f}, bob = bb;
        for (int r = t; r < ld; r += kResThreads) {
          bb = df_fma(bn[r], bn[r], bb);
          bob = df_fma(bn[r], bo[r], bob);
        }
        block_pairs(bb, bob);                      // its barrier publishes bn, bo, bad
        if (bad[1]) { dead = true; break; }
        columns(k, ck, bb, bob);
        __syncthreads();
        if (K == 1) {                              // the next step's row is c_1'
          if (send && w == kResWarps - 1) send_cc(cnew, step + 1);
          update(cnew, step + 1, send, last, r2);
          __syncthreads();
          for (int c = t; c < nc; c += kResThreads) crow(0)[c] = cnew[c];
        } else {
          update(cx, step + 1, send, last, r2);
        }
      } else {
        for (int c = t; c < nc; c += kResThreads) cold[c] = cnew[c] = ck[c];
        __syncthreads();
        if (bad[1]) { dead = true; break; }
        update(cx, step + 1, send, last, r2);
      }
      if (rec) a.tstamp[4 * at + 2] = a.tstamp[4 * at + 3] = globaltimer_ns();
    }
    if (dead) break;
    // objective: the CTAs' sums, in order, in every CTA that needs the value
    df z = df{0.f, 0.f};
    __syncthreads();
    block_pairs(r2, z);
    if (t == 0) {
      st_word(mine + ld + 4 + 2 * (s & 1), r2.h, step);
      st_word(mine + ld + 5 + 2 * (s & 1), r2.l, step);
    }
    bool stop = false;
    const bool need = a.stop_rule != 0 || cta == 0;
    if (need && w == 0) {
      df f2;
      const bool ok = take_pair(ld + 4 + 2 * (s & 1), step, f2);
      if (!ok) bad[2] = 1;
      if (lane == 0) red[2 * kResWarps + 1] = f2;
    }
    if (!inter) {
      // the new B, for the next C step
      for (int i = t; i < K * nrows; i += kResThreads) {
        const int k = i / nrows, r = i - k * nrows;
        __stcg(a.B + (size_t)k * ld + r0 + r, brow[k * rpc + r]);
      }
      ++nbar;
      if (!grid_sync(&a.ctrl->bar, nbar * (unsigned)G, err, tmo)) { dead = true; break; }
    }
    __syncthreads();
    if (bad[2]) { dead = true; break; }
    if (need) {
      const df f2 = red[2 * kResWarps + 1];
      const double f = 0.5 * ((double)f2.h + (double)f2.l);
      if (cta == 0 && t == 0) {
        a.trace[s] = f;
        a.ctrl->sweeps = s + 1;
      }
      if (a.stop_rule == 1) {
        stop = (f == 0.0) || (f_prev > 0.0 && fabs(f_prev - f) / f_prev < a.tol);
      } else if (a.stop_rule == 2) {
        stop = f <= a.tol * a.f0;
      }
      f_prev = f;
    }
    if (stop) {
      if (cta == 0 && t == 0) a.ctrl->stopped = 1;
      break;
    }
  }
  // R and the own rows of B go back (also after an expired wait: B and C
  // are valid then, R is recomputed by the caller)
  __syncthreads();
  if (a.bf16) {
    __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(a.R) + (size_t)j0 * ld;
    for (int i = t; i < nc * ld; i += kResThreads) dst[i] = __float2bfloat16_rn(R[i]);
  } else {
    float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(a.R) + (size_t)j0 * ld);
    for (int i = t; i < nc * ld / 4; i += kResThreads) dst[i] = reinterpret_cast<float4*>(R)[i];
  }
  for (int i = t; i < K * nrows; i += kResThreads) {
    const int k = i / nrows, r = i - k * nrows;
    a.B[(size_t)k * ld + r0 + r] = brow[k * rpc + r];
  }
}

__global__ void __launch_bounds__(kResThreads, 1) resident_kernel(ResArgs a) {
  resident_body(a, blockIdx.x, gridDim.x);
}

// Several instances in one launch, each on its own range of CTAs.
__global__ void __launch_bounds__(kResThreads, 1) resident_multi_kernel(const ResArgs* __restrict__ inst, int ninst) {
  int i = 0;
  while (i + 1 < ninst && (int)blockIdx.x >= inst[i + 1].cta_begin) ++i;
  const ResArgs a = inst[i];
  const int cta = (int)blockIdx.x - a.cta_begin;
  if (cta < 0 || cta >= a.cta_count) return;
  resident_body(a, cta, a.cta_count);
}

// Plan on at most `grid` CTAs: columns dealt evenly; false if they do not fit `budget`.
bool plan_on(int ld, int64_t N, int K, int grid, size_t budget, ResidentPlan* plan) {
  const int64_t nc = (N + grid - 1) / grid;
  if (nc > (1 << 20)) return false;
  const int g = (int)((N + nc - 1) / nc);
  const size_t smem = res_smem(ld, K, (int)nc, g).total;
  if (smem > budget) return false;
  plan->nc = (int)nc;
  plan->grid = g;
  plan->smem = smem;
  plan->words_bytes = (size_t)g * (ld + 8) * sizeof(uint2) + (size_t)ld * sizeof(uint4);
  return true;
}

size_t res_budget(const void* func) {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa{};
  if (cudaFuncGetAttributes(&fa, func) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return (size_t)optin - fa.sharedSizeBytes;
}

ResArgs make_args(const ResidentPlan& plan, const SweepArgs& s, void* words, unsigned step0, bool bf16) {
  ResArgs a{};
  a.R = s.R;
  a.B = s.B;
  a.C = s.C;
  a.Bw = static_cast<uint4*>(words);
  a.Pw = reinterpret_cast<uint2*>(a.Bw + s.ld);
  a.ctrl = s.ctrl;
  a.trace = s.trace;
  a.degen = s.degen;
  a.N = s.N;
  a.ld = s.ld;
  a.K = s.K;
  a.nc = plan.nc;
  a.bf16 = bf16 ? 1 : 0;
  a.n_sweeps = s.n_sweeps;
  a.order = s.order;
  a.step0 = step0;
  a.stop_rule = s.stop_rule;
  a.tol = s.tol;
  a.f_prev = s.f_prev;
  a.f0 = s.f0;
  a.bar_extra = s.bar_extra;
  a.timeout_ns = s.timeout_ns;
  a.tstamp = s.tstamp;
  a.tstamp_cap = s.tstamp_cap;
  a.cta_begin = s.cta_begin;
  a.cta_count = plan.grid;
  return a;
}

}  // namespace

bool plan_resident(int ld, int64_t N, int K, int grid_override, ResidentPlan* plan) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t budget = res_budget((const void*)resident_kernel);
  const int gmax = grid_override > 0 ? std::min(grid_override, sms) : sms;
  // Columns of a CTA: two for each warp (32), the fewest CTAs that gives, so
  // that an exchange has few parties; fewer where a column range must be
  // shorter to fit, more where the grid is at its limit.  A k of 200 x 1000 /
  // 1024 x 2414 / 43 x 1694 in one run: 7.5 / 8.9 / 8.1 us with 8 columns, 6.6 /
  // 8.9 / 7.2 with 16, 6.3 / 8.7 / 6.1 with 32, 7.3 / 8.6 / 6.3 with 64 (GPUs
  // differ by some 5 %, short columns by more).
  ResidentPlan P{};
  for (int nc = 32; nc >= 1 && P.grid == 0; nc /= 2) {
    const int64_t g = (N + nc - 1) / nc;
    if (g > gmax) break;
    plan_on(ld, N, K, (int)g, budget, &P);
  }
  if (P.grid == 0 && !plan_on(ld, N, K, gmax, budget, &P)) return false;
  int per_sm = 0;
  if (cudaFuncSetAttribute(resident_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)budget) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, resident_kernel, kResThreads, P.smem) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    return false;
  }
  *plan = P;
  return true;
}

// Within a launch of several instances the CTAs are shared out by the caller.
size_t resident_multi_budget() { return res_budget((const void*)resident_multi_kernel); }

bool plan_resident_on(size_t budget, int ld, int64_t N, int K, int grid, ResidentPlan* plan) {
  return grid > 0 && plan_on(ld, N, K, grid, budget, plan);
}

cudaError_t launch_resident(const ResidentPlan& plan, const SweepArgs& s, void* words, unsigned step0, bool bf16,
                            cudaStream_t st) {
  ResArgs a = make_args(plan, s, words, step0, bf16);
  a.cta_begin = 0;
  void* params[] = {&a};
  return cudaLaunchCooperativeKernel((const void*)resident_kernel, dim3(plan.grid), dim3(kResThreads), params,
                                     plan.smem, st);
}

size_t resident_args_bytes() { return sizeof(ResArgs); }

void fill_resident_args(void* dst, const ResidentPlan& plan, const SweepArgs& s, void* words, bool bf16) {
  *static_cast<ResArgs*>(dst) = make_args(plan, s, words, 0u, bf16);
}

cudaError_t launch_resident_multi(const void* d_args, int ninst, int grid, size_t smem, cudaStream_t st) {
  const ResArgs* inst = static_cast<const ResArgs*>(d_args);
  const cudaError_t e = cudaFuncSetAttribute(resident_multi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)resident_multi_budget());
  if (e != cudaSuccess) return e;
  void* params[] = {(void*)&inst, (void*)&ninst};
  return cudaLaunchCooperativeKernel((const void*)resident_multi_kernel, dim3(grid), dim3(kResThreads), params, smem, st);
}

}  // namespace did
