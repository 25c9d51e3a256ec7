// Serving runtime: continuous batching of factorisation requests on one GPU.
//
// A worker thread admits queued requests under an HBM budget and a slot
// limit, keeps each active request's X, R, B and C resident, and runs rounds
// that advance every active request by up to `round_sweeps` sweeps.  A
// request's residual decides how (Form):
//   RESIDENT  it fits the SMs' shared memory: such requests are packed into
//             launches, each request on as few CTAs as hold its residual (and
//             more where CTAs are left), because a k of it costs two exchanges
//             whatever the number of CTAs is;
//   DEFER     larger: read-only sweeps on the whole GPU, one request after another,
//             each pass at HBM speed, which a share of the SMs does not reach;
//   PACKED    otherwise (K too large for a short column, or several mid-sized requests at
//             once, pack_mid_sized): the multi-instance sweep kernel, each request on its own
//             CTA range, proportional to its per-sweep work.
// All three stop a request on the device by its own rule.  With every
// request in the multi-instance kernel 24 requests of 20 sweeps took 488 ms;
// see run_round for what they take now.  Between rounds finished requests are retired and new ones
// admitted.  All device memory of a request is one stream-ordered allocation;
// the scratch of the forms is the server's (one request or launch uses it at a
// time), within the budget: it is given back where a request is admitted in
// its place, and a request whose form's scratch does not fit runs PACKED.
#include "did_internal.cuh"

#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <condition_variable>
#include <deque>
#include <map>
#include <mutex>
#include <thread>
#include <vector>

using did::Ctrl;
using did::SweepArgs;

namespace {

constexpr uint64_t kServeTimeoutNs = 4000000000ull;
// Cost model of one column pass of an instance on s CTAs (used to balance a
// round): a fixed part (two grid waits, the b-reduce, the ring's fill) plus
// the residual's read and write at one CTA's share of the HBM bandwidth.
constexpr double kPassFixedS = 12e-6;
constexpr double kCtaBytesPerS = 40e9;
constexpr double kRoundMinS = 5e-3;      // a launch of the multi-instance kernel lasts at least this long
// Costs of a k of a larger request: read-only sweeps alone on the GPU, and the
// multi-instance kernel (the fixed part once, then the read and the write of each request).
constexpr double kDeferFixedS = 20e-6;
constexpr double kDeferBytesPerS = 6.5e12;
constexpr double kPackFixedS = 30e-6;
constexpr double kPackBytesPerS32 = 5.0e12;
constexpr double kPackBytesPerS16 = 4.0e12;
constexpr double kDeferSliceS = 20e-3;   // a larger request's sweeps in one round take at most about this long
// Phase stamps kept per instance (4 per k of its first sweep in a round):
// the measured time of that sweep drives the next round's CTA shares.
constexpr int kStampK = 64;

double now_s(const std::chrono::steady_clock::time_point& t0) {
  return std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
}

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

enum ReqState { QUEUED, ACTIVE, DONE, FAILED };
enum Form { RESIDENT, DEFER, PACKED };

struct Req {
  uint64_t ticket = 0;
  did_request rq{};
  ReqState state = QUEUED;
  did_status status = DID_PENDING;
  int ld = 0;
  size_t bytes = 0;
  bool reserved = false;   // bytes counted in the server's budget ledger
  void* block = nullptr;
  float *X = nullptr, *B = nullptr, *C = nullptr, *P = nullptr, *bold = nullptr;
  void* R = nullptr;
  double *CCp = nullptr, *Sp = nullptr, *OBJp = nullptr;
  int sweeps = 0;
  double cta_s = -1.0;     // measured CTA-seconds per sweep (smoothed); < 0: not measured yet
  int sh_last = 0;         // CTAs of its last round in the multi-instance kernel (0: none, or another form since)
  Form form = PACKED;
  int ctas = 0;            // RESIDENT: fewest CTAs that hold its residual
  did::DeferPlan dplan{};  // DEFER
  std::vector<double> trace;
  std::vector<float> Bh, Ch;   // results on the host after completion
  double t_submit = 0, t_start = 0, t_done = 0;
  bool fetched = false;
};

}  // namespace

struct did_server {
  size_t budget = 0, used = 0, peak = 0;
  bool bf16 = false;
  int max_slots = 1, round_sweeps = 4;
  int dev = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  int grid = 0;
  size_t smem_budget = 0;
  size_t res_budget = 0;             // shared memory of a CTA of the resident kernel on this device
  std::chrono::steady_clock::time_point t0;

  std::mutex mu;
  std::condition_variable cv_work, cv_done;
  std::deque<Req*> queue;
  std::vector<Req*> active;
  std::map<uint64_t, Req*> reqs;
  uint64_t next_ticket = 1;
  bool stopping = false;
  std::thread worker;

  // round scratch (device + pinned host)
  SweepArgs* d_inst = nullptr;
  SweepArgs* h_inst = nullptr;
  Ctrl* d_ctrl = nullptr;
  Ctrl* h_ctrl = nullptr;
  double* d_trace = nullptr;
  double* h_trace = nullptr;
  uint64_t* d_stamp = nullptr;       // [slot][4 kStampK] phase stamps of an instance's first sweep
  uint64_t* h_stamp = nullptr;
  unsigned char* d_res = nullptr;    // [slot] arguments of resident instances
  unsigned char* h_res = nullptr;
  void* scratch = nullptr;           // words of a resident launch, or buffers of a read-only sweep
  size_t scratch_bytes = 0;
  unsigned long long* d_degen = nullptr;
  unsigned long long* d_bad = nullptr;   // negative or non-finite entries of a request's X
  unsigned long long* h_bad = nullptr;
  double* d_part = nullptr;          // dense-pass partial sums
  double* h_part = nullptr;
  int dense_grid = 0;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;

  // statistics
  int64_t submitted = 0, completed = 0, failed = 0, rounds = 0;
  int peak_active = 0;
  double busy_s = 0.0, first_submit = -1.0, last_done = 0.0;
  std::vector<double> latencies;
};

namespace {

// Device bytes of one request (partials sized for the whole grid).
size_t request_bytes(const did_server* s, int64_t M, int64_t N, int K, int ld) {
  const size_t G = (size_t)s->grid;
  size_t b = 0;
  b += a256((size_t)ld * N * 4);                    // X
  b += a256((size_t)ld * N * (s->bf16 ? 2 : 4));    // R
  b += a256((size_t)ld * K * 4);                    // B
  b += a256((size_t)K * N * 4);                     // C
  b += a256(G * ld * 4);                            // P
  b += 3 * a256(G * 2 * 8);                         // CCp, Sp, OBJp
  b += a256((size_t)ld * 4);                        // bold
  (void)M;
  return b;
}

void choose_form(const did_server* s, Req* r);

void free_scratch(did_server* s) {
  if (s->scratch) cudaFreeAsync(s->scratch, s->stream);
  s->scratch = nullptr;
  s->scratch_bytes = 0;
}

// The server's scratch, at least `bytes`; false if the budget (which it shares
// with the requests) or the device has no room for it.
bool need_scratch(did_server* s, size_t bytes) {
  if (bytes <= s->scratch_bytes) return true;
  if (s->used + bytes > s->budget) return false;
  free_scratch(s);
  if (cudaMallocAsync(&s->scratch, bytes, s->stream) != cudaSuccess) {
    cudaGetLastError();
    s->scratch = nullptr;
    return false;
  }
  s->scratch_bytes = bytes;
  return true;
}

// Allocate, generate or copy X, draw the start point and form R = X - B C.
did_status admit(did_server* s, Req* r) {
  const int64_t M = r->rq.M, N = r->rq.N;
  const int K = r->rq.K;
  const int ld = r->ld;
  cudaStream_t st = s->stream;
  cudaError_t got = cudaMallocAsync(&r->block, r->bytes, st);
  if (got != cudaSuccess && s->scratch) {     // the scratch gives way to a request
    cudaGetLastError();
    free_scratch(s);
    got = cudaStreamSynchronize(st);
    if (got == cudaSuccess) got = cudaMallocAsync(&r->block, r->bytes, st);
  }
  if (got != cudaSuccess) {
    cudaGetLastError();
    r->block = nullptr;
    return DID_ENOMEM;
  }
  unsigned char* p = static_cast<unsigned char*>(r->block);
  auto take = [&](size_t n) { void* q = p; p += a256(n); return q; };
  const size_t G = (size_t)s->grid;
  r->X = (float*)take((size_t)ld * N * 4);
  r->R = take((size_t)ld * N * (s->bf16 ? 2 : 4));
  r->B = (float*)take((size_t)ld * K * 4);
  r->C = (float*)take((size_t)K * N * 4);
  r->P = (float*)take(G * ld * 4);
  r->CCp = (double*)take(G * 2 * 8);
  r->Sp = (double*)take(G * 2 * 8);
  r->OBJp = (double*)take(G * 2 * 8);
  r->bold = (float*)take((size_t)ld * 4);

  cudaError_t e = cudaSuccess;
  if (r->rq.X) {
    e = cudaMemcpy2DAsync(r->X, (size_t)ld * 4, r->rq.X, (size_t)M * 4, (size_t)M * 4, (size_t)N,
                          cudaMemcpyDefault, st);
  } else {
    // planted X = B0 C0 + 0.01 |N(0,1)|; B0 and C0 borrow the B and C regions
    e = did::launch_gen_uniform(r->B, M * K, r->rq.seed, 0, st);
    if (e == cudaSuccess) e = did::launch_gen_uniform(r->C, (int64_t)K * N, r->rq.seed, 1, st);
    if (e == cudaSuccess)
      e = did::launch_gen_planted_x_ld(r->X, ld, r->B, r->C, (int)M, N, K, r->rq.seed, 0.01, 0.0, 5.0, st);
  }
  if (e == cudaSuccess && ld > M)
    e = cudaMemset2DAsync(r->X + M, (size_t)ld * 4, 0, (size_t)(ld - M) * 4, (size_t)N, st);
  // a caller's X must be finite and >= 0, as for did_create
  if (e == cudaSuccess && r->rq.X) e = cudaMemsetAsync(s->d_bad, 0, sizeof(unsigned long long), st);
  if (e == cudaSuccess && r->rq.X) e = did::launch_check_nonneg_finite(r->X, (int)M, ld, N, s->d_bad, st);
  if (e == cudaSuccess && r->rq.X)
    e = cudaMemcpyAsync(s->h_bad, s->d_bad, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = did::launch_gen_uniform_padded(r->B, (int)M, ld, K, r->rq.seed, 4, st);
  if (e == cudaSuccess) e = did::launch_gen_uniform(r->C, (int64_t)K * N, r->rq.seed, 5, st);
  if (e == cudaSuccess) {
    did::DenseArgs d{};
    d.X = r->X;
    d.R = r->R;
    d.B = r->B;
    d.C = r->C;
    d.part = s->d_part;
    d.M = (int)M;
    d.ld = ld;
    d.K = K;
    d.N = N;
    d.mode = 0;
    d.bf16 = s->bf16 ? 1 : 0;
    e = did::launch_dense(d, st);
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(s->h_part, s->d_part, sizeof(double) * 3 * s->dense_grid, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return DID_ECUDA;
  }
  if (r->rq.X && *s->h_bad != 0) return DID_EINVAL;
  choose_form(s, r);
  double f = 0.0;
  for (int i = 0; i < s->dense_grid; ++i) f += s->h_part[3 * i];
  r->trace.assign(1, 0.5 * f);
  return DID_OK;
}

// Give back a request's device memory and its share of the budget.  The
// share is returned even when the allocation itself failed (admission
// reserves it before allocating), so a failed admission never shrinks the
// budget left for the requests behind it.
void release(did_server* s, Req* r) {
  if (r->block) {
    cudaFreeAsync(r->block, s->stream);
    r->block = nullptr;
  }
  if (r->reserved) {
    s->used -= r->bytes;
    r->reserved = false;
  }
}

// CTA-seconds one sweep of a request takes: measured in earlier rounds, else
// from the cost model at one CTA (its column passes' bytes at one CTA's share
// of the bandwidth, plus the fixed part of each pass).
double sweep_cta_s(const did_server* s, const Req* r) {
  if (r->cta_s > 0.0) return r->cta_s;
  const double pass_bytes = 2.0 * (double)r->ld * (double)r->rq.N * (s->bf16 ? 2.0 : 4.0);
  return (double)r->rq.K * (kPassFixedS + pass_bytes / kCtaBytesPerS);
}

// Split the launch's CTAs among the active requests so that the slowest
// sweep is as short as possible (a round waits for its slowest instance):
// every request starts with one CTA, and each further CTA goes to the request
// whose sweep, at its CTA-seconds / CTAs, would take longest (ties to the
// lower index).  An instance never gets more CTAs than it has columns.
std::vector<int> shares(const did_server* s, const std::vector<Req*>& act) {
  const int n = (int)act.size();
  std::vector<int> sh(n, 1);
  std::vector<double> w(n);
  for (int i = 0; i < n; ++i) w[i] = sweep_cta_s(s, act[i]);
  for (int left = s->grid - n; left > 0; --left) {
    int best = -1;
    double tb = -1.0;
    for (int i = 0; i < n; ++i) {
      if (sh[i] >= act[i]->rq.N) continue;
      const double t = w[i] / sh[i];
      if (t > tb) { tb = t; best = i; }
    }
    if (best < 0) break;
    ++sh[best];
  }
  return sh;
}

// How a request is swept (see the head of this file).
void choose_form(const did_server* s, Req* r) {
  const int64_t N = r->rq.N;
  const int K = r->rq.K;
  did::ResidentPlan p{};
  r->form = PACKED;
  if (did::plan_resident_on(s->res_budget, r->ld, N, K, s->grid, &p)) {
    int lo = 1, hi = s->grid;
    while (lo < hi) {
      const int mid = (lo + hi) / 2;
      if (did::plan_resident_on(s->res_budget, r->ld, N, K, mid, &p)) hi = mid; else lo = mid + 1;
    }
    r->form = RESIDENT;
    r->ctas = did::plan_resident_on(s->res_budget, r->ld, N, K, lo, &p) ? lo : s->grid;
  } else if (r->ld >= 4 * K && did::plan_defer(r->ld, N, K, s->bf16, 0, &r->dplan)) {
    r->form = DEFER;
  }
}

// Buffers of a read-only sweep of r in the scratch (or, with base null, their size).
struct DeferScratch {
  did::DeferBuffers b{};
  void* tc_ws = nullptr;
  double* part = nullptr;
  size_t bytes = 0;
};
DeferScratch defer_scratch(const did_server* s, const Req* r, unsigned char* base) {
  DeferScratch d;
  const size_t N = (size_t)r->rq.N, K = (size_t)r->rq.K, ld = (size_t)r->ld;
  const size_t G = (size_t)did::refresh_tc_grid();
  size_t o = 0;
  auto take = [&](size_t n) { void* q = base ? base + o : nullptr; o += a256(n); return q; };
  d.b.Bo = (float*)take(ld * K * 4);
  d.b.Co = (float*)take(K * N * 4);
  d.b.T = (float*)take(N * (size_t)(r->dplan.GS / 32) * 4);
  d.b.corr = take(N * 8);
  d.b.P = (float*)take(std::max<size_t>((size_t)r->dplan.npart, 2 * G) * ld * 4);
  d.b.CC0 = (double*)take(2 * G * 8);
  d.b.Xp = take(did::defer_pair_bytes((int)K, r->dplan.grid));
  d.b.Yp = take(did::defer_pair_bytes((int)K, r->dplan.grid));
  d.b.work = (unsigned*)take((K + 1) * 4);
  d.part = (double*)take(G * 8);
  if (did::refresh_tc_supported((int)K, !s->bf16))
    d.tc_ws = take(did::refresh_tc_workspace_bytes((int)r->rq.M, r->ld, r->rq.N, (int)K, !s->bf16));
  d.bytes = o;
  d.b.R = r->R;
  d.b.B = r->B;
  d.b.C = r->C;
  return d;
}

// Common arguments of an instance in slot i.
SweepArgs slot_args(const did_server* s, const Req* r, int i, int n_sweeps) {
  SweepArgs a{};
  a.R = r->R;
  a.B = r->B;
  a.C = r->C;
  a.P = r->P;
  a.CCp = r->CCp;
  a.Sp = r->Sp;
  a.OBJp = r->OBJp;
  a.bold = r->bold;
  a.ctrl = s->d_ctrl + i;
  a.trace = s->d_trace + (size_t)i * s->round_sweeps;
  a.degen = s->d_degen + i;
  a.N = r->rq.N;
  a.M = (int)r->rq.M;
  a.ld = r->ld;
  a.K = r->rq.K;
  a.n_sweeps = n_sweeps;
  a.f_prev = r->trace.back();
  a.f0 = r->trace.front();
  a.stop_rule = r->rq.tol > 0.0 ? 1 : 0;
  a.tol = r->rq.tol;
  a.order = DID_ORDER_INTERLEAVED;
  a.timeout_ns = kServeTimeoutNs;
  return a;
}

// PACKED requests (slots idx of act): one launch of the multi-instance kernel.
cudaError_t launch_packed(did_server* s, const std::vector<Req*>& act, const std::vector<int>& idx) {
  const int n = (int)idx.size();
  std::vector<Req*> sub(n);
  for (int q = 0; q < n; ++q) sub[q] = act[idx[q]];
  const std::vector<int> sh = shares(s, sub);
  // Sweeps per instance: the launch lasts about as long as the slowest
  // instance's single sweep (at least kRoundMinS); faster instances run more
  // sweeps in that time, so no CTA range idles for long.  A sweep's time on
  // sh CTAs is taken as its CTA-seconds / sh.
  std::vector<double> tsw(n);
  double T = kRoundMinS;
  for (int q = 0; q < n; ++q) {
    tsw[q] = sweep_cta_s(s, sub[q]) / (double)sh[q];
    T = std::max(T, tsw[q]);
  }
  size_t smem = 0;
  int begin = 0;
  for (int q = 0; q < n; ++q) {
    Req* r = sub[q];
    const int i = idx[q];
    const int left = r->rq.max_iter - r->sweeps;
    const int nsw = std::max(1, std::min(std::min(s->round_sweeps, left), (int)(T / tsw[q])));
    did::SweepPlan plan{};
    if (did::plan_instance(r->ld, r->rq.N, s->bf16, sh[q], s->smem_budget, &plan) != DID_OK) return cudaErrorInvalidValue;
    smem = std::max(smem, plan.smem);
    SweepArgs a = slot_args(s, r, i, nsw);
    a.GS = plan.GS;
    a.NG = plan.NG;
    a.D = plan.D;
    a.units = plan.units;
    a.nunits = plan.nunits;
    a.dynamic = 0;
    a.npart = plan.npart;
    // the partials of R c_1^T left by the last sweep are valid while the
    // instance keeps its CTA range size (same plan); else a prologue pass
    a.prologue = sh[q] != r->sh_last ? 1 : 0;
    r->sh_last = sh[q];
    a.tstamp = s->d_stamp + (size_t)i * 4 * kStampK;
    a.tstamp_cap = std::min(r->rq.K, kStampK);
    a.pair = plan.pair;
    a.cta_begin = begin;
    a.cta_count = sh[q];
    begin += sh[q];
    s->h_inst[q] = a;
  }
  const cudaError_t e =
      cudaMemcpyAsync(s->d_inst, s->h_inst, sizeof(SweepArgs) * n, cudaMemcpyHostToDevice, s->stream);
  if (e != cudaSuccess) return e;
  return did::launch_sweep_multi(s->bf16, s->d_inst, n, begin, smem, s->stream);
}

// Time of one k of a resident instance in microseconds, as measured on
// launches of one instance (6.3 at 208 rows x 32 columns a CTA, 8.7 at 1024 x
// 32, 12.8 at 2000 x 20, 15.4 at 4112 x 10).
double resident_k_us(int ld, int nc) { return 5.0 + 1.5e-3 * ld + 8e-5 * (double)ld * nc; }

struct Bin {
  std::vector<int> slots;
  std::vector<did::ResidentPlan> plans;
  size_t words = 0;
  int ctas = 0;
};

// RESIDENT requests dealt to launches: longest first into the first launch
// with room, then the CTAs left in a launch go to its slowest instance.
std::vector<Bin> pack(const did_server* s, const std::vector<Req*>& act, std::vector<int> idx) {
  auto cols = [&](int i, int g) { return (int)((act[i]->rq.N + g - 1) / g); };
  auto cost = [&](int i, int g) { return act[i]->rq.K * resident_k_us(act[i]->ld, cols(i, g)); };
  std::sort(idx.begin(), idx.end(), [&](int x, int y) {
    const double a = cost(x, act[x]->ctas), b = cost(y, act[y]->ctas);
    return a != b ? a > b : x < y;
  });
  std::vector<Bin> bins;
  for (int i : idx) {
    size_t q = 0;
    while (q < bins.size() && bins[q].ctas + act[i]->ctas > s->grid) ++q;
    if (q == bins.size()) bins.emplace_back();
    bins[q].slots.push_back(i);
    bins[q].ctas += act[i]->ctas;
  }
  for (Bin& b : bins) {
    const int n = (int)b.slots.size();
    std::vector<int> g(n);
    std::vector<char> full(n, 0);
    for (int q = 0; q < n; ++q) g[q] = act[b.slots[q]]->ctas;
    int left = s->grid - b.ctas;
    while (left > 0) {
      int best = -1;
      for (int q = 0; q < n; ++q)
        if (!full[q] && (best < 0 || cost(b.slots[q], g[q]) > cost(b.slots[best], g[best]))) best = q;
      if (best < 0) break;
      // the next size that shortens its column ranges, while they are wider than one column a warp
      const int nc = cols(b.slots[best], g[best]);
      const int64_t N = act[b.slots[best]]->rq.N;
      const int to = nc > 16 ? (int)((N + nc - 2) / (nc - 1)) : 0;
      if (to == 0 || to - g[best] > left) {
        full[best] = 1;
        continue;
      }
      left -= to - g[best];
      g[best] = to;
    }
    b.ctas = 0;
    for (int q = 0; q < n; ++q) {
      const Req* r = act[b.slots[q]];
      did::ResidentPlan p{};
      if (!did::plan_resident_on(s->res_budget, r->ld, r->rq.N, r->rq.K, g[q], &p))
        did::plan_resident_on(s->res_budget, r->ld, r->rq.N, r->rq.K, r->ctas, &p);
      b.plans.push_back(p);
      b.words += a256(p.words_bytes);
      b.ctas += p.grid;
    }
  }
  return bins;
}

// DEFER requests of this round that take less of the GPU's time in the
// multi-instance kernel: alone each pays about kDeferFixedS a k, whatever its
// size is, and its refresh; together they pay one kPackFixedS a k, then the read
// and the write of their residuals.  The smallest go first, as many as make the
// sum shortest.  A request may change its form between rounds: R is current
// after each.  Measured on 128 requests (64..4096 rows, 256..65536 columns, K 8
// to 64, 64 at once, 300 sweeps each): float32 7.85 solves/s with all of
// them alone, 9.08 so (8.2 with the rates of the model 0.6 and 1.6 times these);
// bfloat16 9.1 and 11.8 (11.4, 11.7); in the multi-instance kernel 6.9 and 9.8.
void pack_mid_sized(const did_server* s, const std::vector<Req*>& act, std::vector<int>* def, std::vector<int>* packed) {
  auto bytes = [&](int i) { return (double)act[i]->ld * (double)act[i]->rq.N * (s->bf16 ? 2.0 : 4.0); };
  auto alone = [&](int i) {
    return act[i]->rq.K * (kDeferFixedS + bytes(i) / kDeferBytesPerS) + (s->bf16 ? 3.0 : 2.0) * bytes(i) / kDeferBytesPerS;
  };
  const double rate = s->bf16 ? kPackBytesPerS16 : kPackBytesPerS32;
  double fixed = 0.0, moved = 0.0, rest = 0.0;
  auto add = [&](int i) {
    fixed = std::max(fixed, act[i]->rq.K * kPackFixedS);
    moved += act[i]->rq.K * 2.0 * bytes(i) / rate;
  };
  std::sort(def->begin(), def->end(), [&](int a, int b) { return bytes(a) != bytes(b) ? bytes(a) < bytes(b) : a < b; });
  for (int i : *packed) add(i);
  for (int i : *def) rest += alone(i);
  size_t take = 0;
  double best = fixed + moved + rest;
  for (size_t q = 0; q < def->size() && packed->size() + q < (size_t)s->grid; ++q) {
    add((*def)[q]);
    rest -= alone((*def)[q]);
    if (fixed + moved + rest < best) {
      best = fixed + moved + rest;
      take = q + 1;
    }
  }
  packed->insert(packed->end(), def->begin(), def->begin() + take);
  def->erase(def->begin(), def->begin() + take);
}

// One round over the active requests; returns false on a CUDA error.
// Measured: 24 requests (64..4096 rows, 256..65536 columns, K 8 to 64, float32)
// of 20 sweeps each: 488 ms with every request in the multi-instance kernel,
// 306 ms with the three forms.
bool run_round(did_server* s, std::vector<Req*>& act) {
  const int n = (int)act.size();
  std::vector<int> res, def, packed;
  for (int i = 0; i < n; ++i) (act[i]->form == RESIDENT ? res : act[i]->form == DEFER ? def : packed).push_back(i);
  pack_mid_sized(s, act, &def, &packed);
  std::vector<Bin> bins = pack(s, act, res);
  // Requests whose form's scratch has no room in the budget beside the requests run PACKED.
  const size_t room = s->budget - s->used;
  size_t scratch = 0;
  for (size_t q = 0; q < bins.size();) {
    if (bins[q].words > room) {
      packed.insert(packed.end(), bins[q].slots.begin(), bins[q].slots.end());
      bins.erase(bins.begin() + q);
    } else {
      scratch = std::max(scratch, bins[q++].words);
    }
  }
  for (size_t q = 0; q < def.size();) {
    const size_t need = defer_scratch(s, act[def[q]], nullptr).bytes;
    if (need > room) {
      packed.push_back(def[q]);
      def.erase(def.begin() + q);
    } else {
      scratch = std::max(scratch, need);
      ++q;
    }
  }
  if (!need_scratch(s, scratch)) {       // no such memory on the device: all of them
    packed.resize(n);
    for (int i = 0; i < n; ++i) packed[i] = i;
    bins.clear();
    def.clear();
  }
  cudaStream_t st = s->stream;
  unsigned char* base = static_cast<unsigned char*>(s->scratch);
  cudaError_t e = cudaMemsetAsync(s->d_ctrl, 0, sizeof(Ctrl) * n, st);
  if (e == cudaSuccess) e = cudaEventRecord(s->ev0, st);
  if (e == cudaSuccess && !packed.empty()) e = launch_packed(s, act, packed);
  // RESIDENT: a launch per bin
  const size_t ab = did::resident_args_bytes();
  int at = 0;
  for (Bin& b : bins) {
    size_t words = 0, smem = 0;
    int begin = 0;
    for (size_t q = 0; q < b.slots.size(); ++q) {
      Req* r = act[b.slots[q]];
      SweepArgs a = slot_args(s, r, b.slots[q], std::min(s->round_sweeps, r->rq.max_iter - r->sweeps));
      a.cta_begin = begin;
      did::fill_resident_args(s->h_res + (at + q) * ab, b.plans[q], a, base + words, s->bf16);
      r->sh_last = 0;
      begin += b.plans[q].grid;
      words += a256(b.plans[q].words_bytes);
      smem = std::max(smem, b.plans[q].smem);
    }
    const int m = (int)b.slots.size();
    if (e == cudaSuccess) e = cudaMemsetAsync(base, 0, words, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(s->d_res + at * ab, s->h_res + at * ab, ab * m, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = did::launch_resident_multi(s->d_res + at * ab, m, begin, smem, st);
    at += m;
  }
  // DEFER: one after another on the whole GPU
  const int G = did::refresh_tc_grid();
  for (int i : def) {
    Req* r = act[i];
    DeferScratch d = defer_scratch(s, r, base);
    d.b.ctrl = s->d_ctrl + i;
    d.b.degen = s->d_degen + i;
    r->sh_last = 0;
    const double sweep_s =
        r->rq.K * (kDeferFixedS + (double)r->ld * r->rq.N * (s->bf16 ? 2.0 : 4.0) / kDeferBytesPerS);
    const int nsw = std::max(1, std::min(std::min(s->round_sweeps, r->rq.max_iter - r->sweeps), (int)(kDeferSliceS / sweep_s)));
    double* tr = s->d_trace + (size_t)i * s->round_sweeps;
    did::DenseArgs da{};
    da.X = r->X;
    da.R = r->R;
    da.B = r->B;
    da.C = r->C;
    da.part = s->d_part;
    da.M = (int)r->rq.M;
    da.ld = r->ld;
    da.K = r->rq.K;
    da.N = r->rq.N;
    da.bf16 = s->bf16 ? 1 : 0;
    da.stop = &d.b.ctrl->stopped;
    if (e == cudaSuccess) e = cudaMemsetAsync(d.b.work, 0, sizeof(unsigned) * (r->rq.K + 1), st);
    for (int q = 0; q < nsw && e == cudaSuccess; ++q) {
      // (the partials of c_1 are in the scratch: another request may have used it since)
      e = did::launch_defer(r->dplan, d.b, r->ld, r->rq.N, r->rq.K, q > 0 && d.tc_ws ? 2 * G : 0, 0, kServeTimeoutNs,
                            nullptr, 0, st);
      if (e == cudaSuccess)
        e = d.tc_ws ? did::launch_refresh_tc(r->X, r->R, r->B, r->C, (int)r->rq.M, r->ld, r->rq.N, r->rq.K, d.tc_ws,
                                             d.part, d.b.P, d.b.CC0, &d.b.ctrl->err, kServeTimeoutNs, st, !s->bf16,
                                             &d.b.ctrl->stopped)
                    : did::launch_dense(da, st);
      if (e == cudaSuccess)
        e = did::launch_defer_close(d.tc_ws ? d.part : s->d_part, d.tc_ws ? G : s->dense_grid, d.tc_ws ? 1 : 3,
                                    d.b.ctrl, d.b.work, r->rq.K + 1, tr + q, r->rq.tol > 0.0 ? 1 : 0, r->rq.tol, r->trace.back(),
                                    r->trace.front(), q == 0, st);
    }
  }
  if (e == cudaSuccess) e = cudaEventRecord(s->ev1, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(s->h_ctrl, s->d_ctrl, sizeof(Ctrl) * n, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(s->h_trace, s->d_trace, sizeof(double) * n * s->round_sweeps, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && !packed.empty())
    e = cudaMemcpyAsync(s->h_stamp, s->d_stamp, sizeof(uint64_t) * n * 4 * kStampK, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  // PACKED: the first sweep's time (its first kc k-steps, scaled to K) in CTA-seconds
  for (int i : packed) {
    Req* r = act[i];
    if (s->h_ctrl[i].sweeps < 1 || s->h_ctrl[i].err != 0) continue;
    const int kc = std::min(r->rq.K, kStampK);
    const uint64_t* st4 = s->h_stamp + (size_t)i * 4 * kStampK;
    const uint64_t t0 = st4[0], t1 = st4[4 * (kc - 1) + 3];
    if (t1 <= t0) continue;
    const double cs = (double)(t1 - t0) * 1e-9 * ((double)r->rq.K / kc) * (double)r->sh_last;
    r->cta_s = r->cta_s > 0.0 ? 0.5 * (r->cta_s + cs) : cs;
  }
  float ms = 0.f;
  cudaEventElapsedTime(&ms, s->ev0, s->ev1);
  s->busy_s += ms * 1e-3;
  s->rounds++;
  s->peak_active = std::max(s->peak_active, n);
  return true;
}

void worker_main(did_server* s) {
  cudaSetDevice(s->dev);
  std::unique_lock<std::mutex> lk(s->mu);
  while (true) {
    // admission (FIFO: a request that does not fit blocks the ones behind it)
    while (!s->queue.empty() && (int)s->active.size() < s->max_slots) {
      Req* r = s->queue.front();
      if (s->used + r->bytes > s->budget) break;
      s->queue.pop_front();
      s->used += r->bytes;
      r->reserved = true;
      if (s->used + s->scratch_bytes > s->budget) free_scratch(s);   // a round asks for what then fits
      s->peak = std::max(s->peak, s->used + s->scratch_bytes);
      r->t_start = now_s(s->t0);
      lk.unlock();
      const did_status st = admit(s, r);
      lk.lock();
      if (st != DID_OK) {
        release(s, r);
        r->state = FAILED;
        r->status = st;
        r->t_done = now_s(s->t0);
        s->failed++;
        s->cv_done.notify_all();
        continue;
      }
      r->state = ACTIVE;
      s->active.push_back(r);
    }
    if (s->active.empty()) {
      if (s->stopping && s->queue.empty()) break;
      s->cv_work.wait(lk);
      continue;
    }
    std::vector<Req*> act = s->active;
    lk.unlock();
    const bool ok = run_round(s, act);
    lk.lock();
    s->peak = std::max(s->peak, s->used + s->scratch_bytes);
    const double t = now_s(s->t0);
    std::vector<Req*> still;
    for (int i = 0; i < (int)act.size(); ++i) {
      Req* r = act[i];
      bool finished = false;
      if (!ok || s->h_ctrl[i].err != 0) {
        r->state = FAILED;
        r->status = ok ? DID_ETIMEOUT : DID_ECUDA;
        finished = true;
        s->failed++;
      } else {
        const Ctrl& c = s->h_ctrl[i];
        for (int k = 0; k < c.sweeps; ++k) r->trace.push_back(s->h_trace[(size_t)i * s->round_sweeps + k]);
        r->sweeps += c.sweeps;
        if (c.stopped || r->sweeps >= r->rq.max_iter) {
          r->Bh.resize((size_t)r->rq.M * r->rq.K);
          r->Ch.resize((size_t)r->rq.K * r->rq.N);
          cudaMemcpy2DAsync(r->Bh.data(), (size_t)r->rq.M * 4, r->B, (size_t)r->ld * 4, (size_t)r->rq.M * 4,
                            (size_t)r->rq.K, cudaMemcpyDeviceToHost, s->stream);
          cudaMemcpyAsync(r->Ch.data(), r->C, (size_t)r->rq.K * r->rq.N * 4, cudaMemcpyDeviceToHost, s->stream);
          cudaStreamSynchronize(s->stream);
          r->state = DONE;
          r->status = DID_OK;
          finished = true;
          s->completed++;
          s->latencies.push_back(t - r->t_submit);
          s->last_done = t;
        }
      }
      if (finished) {
        r->t_done = t;
        release(s, r);
      } else {
        still.push_back(r);
      }
    }
    s->active.swap(still);
    s->cv_done.notify_all();
  }
}

void fill_result(const Req* r, did_result* res) {
  if (!res) return;
  res->status = r->state == QUEUED || r->state == ACTIVE ? DID_PENDING : r->status;
  res->iters = r->sweeps;
  res->obj = r->trace.empty() ? 0.0 : r->trace.back();
  res->t_submit = r->t_submit;
  res->t_start = r->t_start;
  res->t_done = r->t_done;
}

}  // namespace

extern "C" {

did_status did_server_create(size_t hbm_budget_bytes, did_precision precision, int32_t max_slots,
                             int32_t round_sweeps, void* stream, did_server** out) {
  if (!out) return DID_EINVAL;
  *out = nullptr;
  if (hbm_budget_bytes == 0 || max_slots < 1 || round_sweeps < 1 || round_sweeps > 64 ||
      (precision != DID_FP32 && precision != DID_BF16R))
    return DID_EINVAL;
  did_server* s = new did_server();
  s->budget = hbm_budget_bytes;
  s->bf16 = precision == DID_BF16R;
  s->round_sweeps = round_sweeps;
  s->t0 = std::chrono::steady_clock::now();
  cudaGetDevice(&s->dev);
  if (did::serve_launch_config(s->bf16, &s->grid, &s->smem_budget) != DID_OK) {
    delete s;
    return DID_ECUDA;
  }
  s->max_slots = std::min(max_slots, s->grid);
  s->res_budget = did::resident_multi_budget();
  s->dense_grid = did::dense_grid();
  bool ok = true;
  if (stream) {
    s->stream = (cudaStream_t)stream;
  } else {
    ok = cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking) == cudaSuccess;
    s->own_stream = true;
  }
  const int S = s->max_slots;
  ok = ok && cudaMalloc(&s->d_inst, sizeof(SweepArgs) * S) == cudaSuccess;
  ok = ok && cudaMallocHost(&s->h_inst, sizeof(SweepArgs) * S) == cudaSuccess;
  ok = ok && cudaMalloc(&s->d_ctrl, sizeof(Ctrl) * S) == cudaSuccess;
  ok = ok && cudaMallocHost(&s->h_ctrl, sizeof(Ctrl) * S) == cudaSuccess;
  ok = ok && cudaMalloc(&s->d_trace, sizeof(double) * S * round_sweeps) == cudaSuccess;
  ok = ok && cudaMallocHost(&s->h_trace, sizeof(double) * S * round_sweeps) == cudaSuccess;
  ok = ok && cudaMalloc(&s->d_stamp, sizeof(uint64_t) * S * 4 * kStampK) == cudaSuccess;
  ok = ok && cudaMallocHost(&s->h_stamp, sizeof(uint64_t) * S * 4 * kStampK) == cudaSuccess;
  ok = ok && cudaMalloc(&s->d_res, did::resident_args_bytes() * S) == cudaSuccess;
  ok = ok && cudaMallocHost(&s->h_res, did::resident_args_bytes() * S) == cudaSuccess;
  ok = ok && cudaMalloc(&s->d_degen, sizeof(unsigned long long) * S) == cudaSuccess;
  ok = ok && cudaMalloc(&s->d_bad, sizeof(unsigned long long)) == cudaSuccess;
  ok = ok && cudaMallocHost(&s->h_bad, sizeof(unsigned long long)) == cudaSuccess;
  ok = ok && cudaMalloc(&s->d_part, sizeof(double) * 3 * s->dense_grid) == cudaSuccess;
  ok = ok && cudaMallocHost(&s->h_part, sizeof(double) * 3 * s->dense_grid) == cudaSuccess;
  ok = ok && cudaEventCreate(&s->ev0) == cudaSuccess && cudaEventCreate(&s->ev1) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    did_server_destroy(s);
    return DID_ENOMEM;
  }
  s->worker = std::thread(worker_main, s);
  *out = s;
  return DID_OK;
}

did_status did_server_submit(did_server* s, const did_request* req, uint64_t* ticket) {
  if (!s || !req || req->M < 1 || req->N < 1 || req->K < 1 || req->K > std::min(req->M, req->N) ||
      req->max_iter < 1 || !(req->tol >= 0.0) || req->M > (1 << 30))
    return DID_EINVAL;
  const int ld = (int)((req->M + 15) / 16 * 16);
  if (ld > did::serve_max_ld(s->bf16)) return DID_E_TOO_LARGE;
  Req* r = new Req();
  r->rq = *req;
  r->ld = ld;
  r->bytes = request_bytes(s, req->M, req->N, req->K, ld);
  if (r->bytes > s->budget) {
    delete r;
    return DID_E_TOO_LARGE;
  }
  std::lock_guard<std::mutex> lk(s->mu);
  r->ticket = s->next_ticket++;
  r->t_submit = now_s(s->t0);
  if (s->first_submit < 0) s->first_submit = r->t_submit;
  s->reqs[r->ticket] = r;
  s->queue.push_back(r);
  s->submitted++;
  if (ticket) *ticket = r->ticket;
  s->cv_work.notify_one();
  return DID_OK;
}

did_status did_server_poll(did_server* s, uint64_t ticket, did_result* res) {
  if (!s) return DID_EINVAL;
  std::lock_guard<std::mutex> lk(s->mu);
  auto it = s->reqs.find(ticket);
  if (it == s->reqs.end()) return DID_EINVAL;
  fill_result(it->second, res);
  const Req* r = it->second;
  return (r->state == QUEUED || r->state == ACTIVE) ? DID_PENDING : r->status;
}

did_status did_server_wait(did_server* s, uint64_t ticket, int32_t timeout_ms, did_result* res) {
  if (!s) return DID_EINVAL;
  std::unique_lock<std::mutex> lk(s->mu);
  auto it = s->reqs.find(ticket);
  if (it == s->reqs.end()) return DID_EINVAL;
  Req* r = it->second;
  auto done = [&] { return r->state == DONE || r->state == FAILED; };
  if (timeout_ms < 0) {
    s->cv_done.wait(lk, done);
  } else if (!s->cv_done.wait_for(lk, std::chrono::milliseconds(timeout_ms), done)) {
    fill_result(r, res);
    return DID_PENDING;
  }
  fill_result(r, res);
  return r->status;
}

did_status did_server_fetch(did_server* s, uint64_t ticket, float* B, float* C) {
  if (!s) return DID_EINVAL;
  std::lock_guard<std::mutex> lk(s->mu);
  auto it = s->reqs.find(ticket);
  if (it == s->reqs.end()) return DID_EINVAL;
  Req* r = it->second;
  if (r->state == QUEUED || r->state == ACTIVE) return DID_PENDING;
  if (r->state == FAILED) return r->status;
  if (r->fetched) return DID_EINVAL;
  if (B && cudaMemcpy(B, r->Bh.data(), r->Bh.size() * 4, cudaMemcpyDefault) != cudaSuccess) {
    cudaGetLastError();
    return DID_ECUDA;
  }
  if (C && cudaMemcpy(C, r->Ch.data(), r->Ch.size() * 4, cudaMemcpyDefault) != cudaSuccess) {
    cudaGetLastError();
    return DID_ECUDA;
  }
  r->fetched = true;
  std::vector<float>().swap(r->Bh);
  std::vector<float>().swap(r->Ch);
  return DID_OK;
}

did_status did_server_stats(did_server* s, did_server_stats_t* out) {
  if (!s || !out) return DID_EINVAL;
  std::lock_guard<std::mutex> lk(s->mu);
  memset(out, 0, sizeof(*out));
  out->submitted = s->submitted;
  out->completed = s->completed;
  out->failed = s->failed;
  out->peak_bytes = s->peak;
  out->peak_active = s->peak_active;
  out->rounds = s->rounds;
  out->busy_s = s->busy_s;
  if (s->completed > 0) {
    std::vector<double> l = s->latencies;
    std::sort(l.begin(), l.end());
    auto pct = [&](double p) {
      const double x = p * (double)(l.size() - 1);
      const size_t i = (size_t)floor(x);
      const double f = x - (double)i;
      return i + 1 < l.size() ? l[i] * (1 - f) + l[i + 1] * f : l[i];
    };
    out->p50_ms = 1e3 * pct(0.50);
    out->p99_ms = 1e3 * pct(0.99);
    const double span = s->last_done - s->first_submit;
    out->solves_per_s = span > 0 ? (double)s->completed / span : 0.0;
  }
  return DID_OK;
}

void did_server_destroy(did_server* s) {
  if (!s) return;
  {
    std::lock_guard<std::mutex> lk(s->mu);
    s->stopping = true;
    s->cv_work.notify_all();
  }
  if (s->worker.joinable()) s->worker.join();
  free_scratch(s);
  if (s->stream) cudaStreamSynchronize(s->stream);
  cudaFree(s->d_res);
  cudaFreeHost(s->h_res);
  for (auto& kv : s->reqs) {
    if (kv.second->block) cudaFree(kv.second->block);
    delete kv.second;
  }
  cudaFree(s->d_inst);
  cudaFreeHost(s->h_inst);
  cudaFree(s->d_ctrl);
  cudaFreeHost(s->h_ctrl);
  cudaFree(s->d_trace);
  cudaFreeHost(s->h_trace);
  cudaFree(s->d_stamp);
  cudaFreeHost(s->h_stamp);
  cudaFree(s->d_degen);
  cudaFree(s->d_bad);
  cudaFreeHost(s->h_bad);
  cudaFree(s->d_part);
  cudaFreeHost(s->h_part);
  if (s->ev0) cudaEventDestroy(s->ev0);
  if (s->ev1) cudaEventDestroy(s->ev1);
  if (s->own_stream && s->stream) cudaStreamDestroy(s->stream);
  delete s;
}

}  // extern "C"
