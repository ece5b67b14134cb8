// libfit: the fused propagate + Kalman-update kernels over runs of same-mode
// events, and the C ABI of fit.h (handle, fit_propagate_update,
// fit_propagate_update_noalloc, fit_sync).  The batched persistent form is in
// batch.cu.
#include <cuda_runtime.h>

#include <chrono>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <string>
#include <thread>
#include <type_traits>

#include "fit.h"
#include "fused.cuh"

namespace fitimpl {

thread_local std::string g_last_error;

int fail(int code, const std::string& msg) {
  g_last_error = msg;
  return code;
}

int cuda_fail(cudaError_t e, const char* what) {
  return fail(FIT_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

namespace {

// The thread's track t: its pair's first one, or a lone one.  The first
// blocks take the lone tracks, so that their one-lane path runs beside the
// pairs of other blocks (in a pair's warp it would run after them: a range
// with odd edges took 38 us instead of 22 at 8191 tracks).  half_part: the
// same for a launch with one thread per track, for the launch's block
// `block`.  (Two functions: one with the block and the tracks per thread as
// parameters made the pairs' kernels 0.8 % slower.)
enum class Part { kNone, kPair, kLone };
template <int K>
__device__ __forceinline__ Part pair_part(const FitArgs& a, const PairRuns<K>& r, int64_t& t) {
  const unsigned lone_blocks = (r.nlone + kBlock - 1) / kBlock;
  if (blockIdx.x < lone_blocks) {
    const unsigned i = blockIdx.x * kBlock + threadIdx.x;
    if (i >= r.nlone) return Part::kNone;
    t = a.t0 + r.lone[i];
    return Part::kLone;
  }
  const unsigned i = (blockIdx.x - lone_blocks) * kBlock + threadIdx.x;
  if (i >= r.pairs.n) return Part::kNone;
  t = a.t0 + run_element(r.pairs, i, 2);
  return Part::kPair;
}
template <int K>
__device__ __forceinline__ Part half_part(int64_t t0, const PairRuns<K>& r, unsigned block,
                                          int64_t& t) {
  const unsigned lone_blocks = (r.nlone + kBlock - 1) / kBlock;
  if (block < lone_blocks) {
    const unsigned i = block * kBlock + threadIdx.x;
    if (i >= r.nlone) return Part::kNone;
    t = t0 + r.lone[i];
    return Part::kLone;
  }
  const unsigned i = (block - lone_blocks) * kBlock + threadIdx.x;
  if (i / 2 >= r.pairs.n) return Part::kNone;
  t = t0 + run_element(r.pairs, i / 2, 2) + (i & 1);
  return Part::kPair;
}
// Blocks of kBlock threads for r's tracks.
template <int TPT, int K>
unsigned part_blocks(const PairRuns<K>& r) {
  return (r.nlone + kBlock - 1) / kBlock + (r.pairs.n * (2 / TPT) + kBlock - 1) / kBlock;
}

// 3 resident blocks per SM for p2r (168 registers, no spills; 2 blocks were
// 17 % slower); p2z fits 4 (127 registers, no spills).  100 events of 9600
// tracks: p2r 242.0 us, p2z 168.0 us, the dependent chains of a layer keeping
// the FP32 pipe 59 and 63 % busy.
template <int MODE, int L, int K>
__global__ void __launch_bounds__(kBlock, MODE == FIT_MODE_Z ? 4 : 3)
    fit_fused_kernel(const __grid_constant__ FitArgs a, const __grid_constant__ PairRuns<K> r) {
  int64_t t;
  const Part part = pair_part(a, r, t);
  if (part == Part::kNone) return;
  unsigned st[2] = {0u, 0u}, iters[2] = {0u, 0u};
  if (part == Part::kPair)
    run_whole_pair<MODE, L, MODE == FIT_MODE_Z && L == 0>(a, a.geo, t, st, iters);
  else
    run_lone<MODE, L>(a, a.geo, t, st[0], iters[0]);
  if (st[0]) count_status(st[0], a.counters);
  if (st[1]) count_status(st[1], a.counters);
  if (MODE == FIT_MODE_R) count_iterations(iters[0] + iters[1], &a.counters[4]);
}

// Adds a track's status and iterations to its event's counters; evt_first
// holds the first track of each of the nevt events.
template <int MODE, class Off>
__device__ __forceinline__ void count_event(const FitArgs& a, int64_t t, unsigned st, unsigned iters,
                                            const Off* __restrict__ evt_first, int nevt) {
  unsigned long long* cnt = a.counters + (int64_t)event_of(t, evt_first, nevt) * kEventSlots + 1;
  if (st) count_status(st, cnt);
  if (MODE == FIT_MODE_R && iters) atomicAdd(&cnt[4], (unsigned long long)iters);
}

template <int MODE, int K>
__global__ void __launch_bounds__(kBlock, MODE == FIT_MODE_Z ? 4 : 3)
    fit_fused_kernel_noalloc(const __grid_constant__ FitArgs a,
                             const __grid_constant__ PairRuns<K> r,
                             const int64_t* __restrict__ evt_off, int nevt) {
  int64_t t;
  const Part part = pair_part(a, r, t);
  if (part == Part::kNone) return;
  unsigned st[2] = {0u, 0u}, iters[2] = {0u, 0u};
  if (part == Part::kPair)
    run_whole_pair<MODE>(a, a.geo, t, st, iters);
  else
    run_lone<MODE>(a, a.geo, t, st[0], iters[0]);
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (i == 0 || part == Part::kPair)
      count_event<MODE>(a, t + i, st[i], iters[i], evt_off, nevt);
}

// The whole of a small call, both modes in one launch and one track per
// thread: with at most one warp per scheduler the layers' dependent chains
// set the time, and a thread's chain is shorter with one track than with two
// (each packed FP32 operation holds the pipe two cycles, and the MUFU and
// control instructions run per track).  1024 tracks: p2r 18.4 -> 12.3 us,
// p2z 14.3 -> 10.3 us, both 18.5 -> 12.3 us, without a second stream's fork
// and join.
template <int K>
struct SmallArgs {
  FitArgs a;  // t0, geo unused
  Geo geo[2];
  int64_t t0[2];
  unsigned blocks_r;  // the p2r events' blocks, then the p2z events'
  PairRuns<K> runs[2];
};

// The first track of each event of a small call, as a kernel parameter.
template <int K>
struct EventTable {
  int n;
  uint32_t first[K];
};
constexpr int kSmallEvents = 256;

// E > 0: count per event (as fit_fused_kernel_noalloc).
template <int L, int E>
__global__ void __launch_bounds__(kBlock)
    fit_small_kernel(const __grid_constant__ SmallArgs<kSmallRuns> s,
                     const __grid_constant__ EventTable<(E > 0 ? E : 1)> ev) {
  auto run = [&](auto mode, unsigned block) {
    constexpr int MODE = decltype(mode)::value;
    int64_t t;
    const Part part = half_part(s.t0[MODE], s.runs[MODE], block, t);
    if (part == Part::kNone) return;
    unsigned st = 0u, iters = 0u;
    if (part == Part::kPair)
      run_half_pair<MODE, L>(s.a, s.geo[MODE], t, st, iters);
    else
      run_lone<MODE, L>(s.a, s.geo[MODE], t, st, iters);
    if constexpr (E > 0) {
      count_event<MODE>(s.a, t, st, iters, ev.first, ev.n);
    } else {
      if (st) count_status(st, s.a.counters);
      if (MODE == FIT_MODE_R) count_iterations(iters, &s.a.counters[4]);
    }
  };
  if (blockIdx.x < s.blocks_r)
    run(std::integral_constant<int, FIT_MODE_R>(), blockIdx.x);
  else
    run(std::integral_constant<int, FIT_MODE_Z>(), blockIdx.x - s.blocks_r);
}

}  // namespace

// Copies the two modes' geometry and numerics into h (no allocation).
int configure_modes(fit_handle* h, const fit_config* cfg_r, const fit_config* cfg_z,
                    const char* who) {
  const fit_config* cfgs[2] = {cfg_r, cfg_z};
  for (int m = 0; m < 2; ++m) {
    const fit_config* c = cfgs[m];
    if (!c) continue;
    if (c->nlayer < 1 || c->nlayer > FIT_MAX_LAYERS || !c->surf)
      return fail(FIT_ERR_ARG, std::string(who) + ": nlayer out of range or surf is NULL");
    for (int l = 0; l < c->nlayer; ++l) {
      if (!(c->surf[l] == c->surf[l]) || (m == FIT_MODE_R && !(c->surf[l] > 0.f)))
        return fail(FIT_ERR_ARG, std::string(who) + ": invalid surface position");
      h->geo[m].surf.s[l] = c->surf[l];
    }
    h->has[m] = true;
    h->nlayer[m] = c->nlayer;
    h->geo[m].kB = fitk::kA * c->B;
    h->B[m] = c->B;
    h->geo[m].max_iter = c->max_iter > 0 ? c->max_iter : 10;
    h->geo[m].tol = c->tol > 0.f ? c->tol : 1e-6f;
    if (c->start != FIT_START_CROSSING && c->start != FIT_START_LINE)
      return fail(FIT_ERR_ARG, std::string(who) + ": start is not a FIT_START_* value");
    h->geo[m].line_start = c->start == FIT_START_LINE;
  }
  return FIT_OK;
}

// Argument checks shared by the entry points that run the fused kernel.
int check_call(const fit_handle* h, const fit_tracks_in* in, const fit_tracks_out* out,
               const fit_hits* hits, int nevt, const int64_t* ntrk, int nlayer,
               const int32_t* mode, int64_t* total_out, const char* who) {
  const std::string w(who);
  if (!in || !out || !hits) return fail(FIT_ERR_ARG, w + ": NULL argument");
  if (nevt < 0) return fail(FIT_ERR_ARG, w + ": nevt < 0");
  if (nevt > 0 && (!ntrk || !mode)) return fail(FIT_ERR_ARG, w + ": ntrk or mode is NULL");
  int64_t total = 0;
  for (int e = 0; e < nevt; ++e) {
    if (ntrk[e] < 0) return fail(FIT_ERR_ARG, w + ": ntrk[e] < 0");
    if (mode[e] != FIT_MODE_R && mode[e] != FIT_MODE_Z)
      return fail(FIT_ERR_ARG, w + ": mode[e] is not FIT_MODE_R or FIT_MODE_Z");
    if (!h->has[mode[e]]) return fail(FIT_ERR_ARG, w + ": mode not configured");
    if (h->nlayer[mode[e]] != nlayer)
      return fail(FIT_ERR_ARG, w + ": nlayer differs from the configured one");
    total += ntrk[e];
  }
  *total_out = total;
  if (total == 0) return FIT_OK;
  if (nlayer < 1 || nlayer > FIT_MAX_LAYERS) return fail(FIT_ERR_ARG, w + ": nlayer out of range");
  if (!in->par || !in->cov || !in->q || !out->par || !out->cov || !out->q || !out->chi2 ||
      !hits->pos || !hits->cov)
    return fail(FIT_ERR_ARG, w + ": NULL data pointer");
  const void* ptrs[] = {in->par, in->cov, in->q, out->par, out->cov, out->q, out->chi2,
                        hits->pos, hits->cov};
  for (const void* p : ptrs)
    if (!aligned16(p)) return fail(FIT_ERR_ARG, w + ": pointer not 16-byte aligned");
  if (in->ld < total || out->ld < total || hits->ld < total)
    return fail(FIT_ERR_ARG, w + ": ld smaller than the number of tracks");
  if ((in->ld | out->ld | hits->ld) & 3) return fail(FIT_ERR_ARG, w + ": ld not a multiple of 4");
  return FIT_OK;
}

FitArgs base_args(const fit_tracks_in* in, const fit_tracks_out* out, const fit_hits* hits,
                  int nlayer, unsigned long long* counters) {
  FitArgs a{};
  a.par_in = in->par;
  a.cov_in = in->cov;
  a.q_in = in->q;
  a.ld_in = in->ld;
  a.par_out = out->par;
  a.cov_out = out->cov;
  a.q_out = out->q;
  a.chi2 = out->chi2;
  a.chi2_layer = out->chi2_layer;
  a.status = out->status;
  a.ld_out = out->ld;
  a.hpos = hits->pos;
  a.hcov = hits->cov;
  a.ld_hit = hits->ld;
  a.nlayer = nlayer;
  a.counters = counters;
  return a;
}

// Adds the tracks [t0, t1) (relative to the launch's even base) to r.
void add_run(PairRuns<kMaxRuns>& r, uint32_t t0, uint32_t t1) {
  const uint32_t p0 = (t0 + 1) & ~1u, p1 = t1 & ~1u;
  if (t0 & 1) r.lone[r.nlone++] = t0;
  if (p1 > p0) {
    Runs<kMaxRuns>& p = r.pairs;
    p.first[p.nrun] = p0;
    p.before[p.nrun++] = p.n;
    p.n += (p1 - p0) / 2;
  }
  if ((t1 & 1) && t1 > p0) r.lone[r.nlone++] = t1 - 1;
}

// The events' tracks as one launch per mode: the runs of consecutive
// same-mode events gathered in a table, with a new launch where it is full
// or its tracks span 2^31.  launch(a, m, r) issues the kernel for the
// runs r of mode m (a.t0: their base; a.geo: the mode's geometry).
// An uneven mixed batch (500 events, 1M tracks, ~250 runs) takes 0.219 ms in
// two launches; with one launch per run it took 4.11 ms, a run's few blocks
// leaving most SMs idle for the ~20 us of its layers.
// by_event: every event is a run of its own.
template <class Launch>
int launch_runs(const fit_handle* h, FitArgs a, bool by_event, int nevt, const int64_t* ntrk,
                const int32_t* mode, const char* who, Launch launch) {
  for (int m : {FIT_MODE_R, FIT_MODE_Z}) {
    PairRuns<kMaxRuns> r;
    auto clear = [&r]() { r.pairs.nrun = 0, r.pairs.n = 0, r.nlone = 0; };
    clear();
    auto flush = [&]() {
      if (!r.pairs.n && !r.nlone) return FIT_OK;
      launch(a, m, r);
      clear();
      cudaError_t err = cudaGetLastError();
      return err == cudaSuccess ? FIT_OK : cuda_fail(err, (std::string(who) + ": launch").c_str());
    };
    a.geo = h->geo[m];
    a.t0 = 0;
    constexpr int64_t kSpan = int64_t(1) << 31;
    int64_t t = 0;
    for (int e = 0; e < nevt;) {
      if (mode[e] != m) {
        t += ntrk[e++];
        continue;
      }
      int64_t t1 = t + ntrk[e++];
      while (!by_event && e < nevt && mode[e] == m) t1 += ntrk[e++];
      while (t < t1) {
        if (!r.pairs.nrun && !r.nlone) a.t0 = t & ~int64_t(1);
        const int64_t end = a.t0 + kSpan < t1 ? a.t0 + kSpan : t1;  // (even where it cuts a run)
        if (r.pairs.nrun == kMaxRuns || r.nlone + 2 > 2 * kMaxRuns || end <= t) {
          const int rc = flush();
          if (rc != FIT_OK) return rc;
          continue;
        }
        add_run(r, (uint32_t)(t - a.t0), (uint32_t)(end - a.t0));
        t = end;
      }
      t = t1;
    }
    const int rc = flush();
    if (rc != FIT_OK) return rc;
  }
  return FIT_OK;
}

// Copies r into a table of K runs, if it fits.
template <int K>
bool copy_table(const PairRuns<kMaxRuns>& r, PairRuns<K>& to) {
  if (r.pairs.nrun > K || r.nlone > 2 * K) return false;
  to.pairs.nrun = r.pairs.nrun;
  to.pairs.n = r.pairs.n;
  to.nlone = r.nlone;
  to.pairs.first[0] = to.pairs.before[0] = 0;
  std::memcpy(to.pairs.first, r.pairs.first, r.pairs.nrun * sizeof(uint32_t));
  std::memcpy(to.pairs.before, r.pairs.before, r.pairs.nrun * sizeof(uint32_t));
  std::memcpy(to.lone, r.lone, r.nlone * sizeof(uint32_t));
  return true;
}

// Shared memory of an SM is split from its L1 cache, and an SM holds blocks of
// two kernels at once only if both ask for the same split.  p2z stages its
// hits (10 KiB a block, four blocks an SM: a split of 64 KiB); the p2r launch
// beside it, which has no use for shared memory, asks for as much (three
// blocks an SM).  Without it the p2z launch waits for SMs to run empty: 40000
// tracks of each mode 49.0 us, the sum of the two, instead of 34.5; 100 events
// of 9600 of each 400.6 instead of 395.0; p2r alone the same.
template <int MODE, int L>
constexpr unsigned kSplitBytes = MODE == FIT_MODE_R && L == 0 ? 13 * 1024 : 0;

template <int MODE, int L>
void launch_fused(const FitArgs& a, const PairRuns<kMaxRuns>& r, cudaStream_t s) {
  constexpr unsigned smem = kSplitBytes<MODE, L>;
  PairRuns<1> one;
  if (copy_table(r, one))
    fit_fused_kernel<MODE, L, 1><<<part_blocks<2>(one), kBlock, smem, s>>>(a, one);
  else
    fit_fused_kernel<MODE, L, kMaxRuns><<<part_blocks<2>(r), kBlock, smem, s>>>(a, r);
}

// The events as one launch of fit_small_kernel: launch(args, blocks) issues
// it.  Returns false, with nothing launched, if their runs do not fit its
// tables.
template <class Launch>
bool launch_small(const fit_handle* h, const FitArgs& a, bool by_event, int nevt,
                  const int64_t* ntrk, const int32_t* mode, Launch launch) {
  SmallArgs<kSmallRuns> s;
  s.a = a;
  unsigned blocks[2] = {0, 0};
  int tables[2] = {0, 0};
  bool fits = true;
  for (int m = 0; m < 2; ++m) {
    s.geo[m] = h->geo[m];
    s.t0[m] = 0;
    s.runs[m].pairs.nrun = 0, s.runs[m].pairs.n = 0, s.runs[m].nlone = 0;
  }
  const int rc = launch_runs(h, a, by_event, nevt, ntrk, mode, "fit_small",
                             [&](const FitArgs& a1, int m, const PairRuns<kMaxRuns>& r) {
                               fits = fits && tables[m]++ == 0 && copy_table(r, s.runs[m]);
                               s.t0[m] = a1.t0;
                               blocks[m] = part_blocks<1>(r);
                             });
  if (rc != FIT_OK || !fits) return false;
  s.blocks_r = blocks[FIT_MODE_R];
  launch(s, blocks[0] + blocks[1]);
  return true;
}

// A call is small where one track per thread leaves every scheduler at most
// one warp (a block of 128 per SM, 19456 tracks): 8192 p2r tracks take 14.3 us
// in the small kernel and 18.5 in pairs.  With two warps per scheduler, at
// 32768 tracks, pairs are as fast (18.5 us), at 65536 faster (26.6 against 28.3).
static bool is_small(int sms, int64_t call_tracks) { return call_tracks <= (int64_t)sms * kBlock; }
static bool is_small(const fit_handle* h, int64_t call_tracks) { return is_small(h->sms, call_tracks); }

// The fused fit of events [0, nevt) on the tracks of a.
int run_fit(const fit_handle* h, const FitArgs& a, const RunOptions& o, int nevt,
            const int64_t* ntrk, const int32_t* mode, const char* who, ModeStreams& ms) {
  const bool soa = o.layout == FIT_LAYOUT_SOA;
  const cudaStream_t s = ms.of(FIT_MODE_R);
  if (!o.seeded && is_small(h, o.call_tracks)) {
    const bool done = launch_small(h, a, o.by_event, nevt, ntrk, mode,
                                   [&](const auto& args, unsigned nblk) {
                                     if (soa)
                                       fit_small_kernel<0, 0><<<nblk, kBlock, 0, s>>>(args, {});
                                     else
                                       fit_small_kernel<1, 0><<<nblk, kBlock, 0, s>>>(args, {});
                                   });
    if (done) {
      const cudaError_t e = cudaGetLastError();
      return e == cudaSuccess ? FIT_OK : cuda_fail(e, (std::string(who) + ": launch").c_str());
    }
  }
  if (o.seeded) {
    const int rc = launch_seeded_fit(h, a, nevt, ntrk, mode, who, s);
    if (rc != FIT_OK) return rc;
  }
  return launch_runs(h, a, o.by_event, nevt, ntrk, mode, who,
                     [&](const FitArgs& a1, int m, const PairRuns<kMaxRuns>& r) {
                       if (m == FIT_MODE_R && o.seeded) return;
                       const cudaStream_t sm = ms.of(m);
                       if (soa)
                         m == FIT_MODE_Z ? launch_fused<FIT_MODE_Z, 0>(a1, r, sm)
                                         : launch_fused<FIT_MODE_R, 0>(a1, r, sm);
                       else
                         m == FIT_MODE_Z ? launch_fused<FIT_MODE_Z, 1>(a1, r, sm)
                                         : launch_fused<FIT_MODE_R, 1>(a1, r, sm);
                     });
}

cudaError_t create_side(SideStream& x) {
  cudaError_t e = cudaStreamCreateWithFlags(&x.st, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&x.fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&x.join, cudaEventDisableTiming);
  if (e != cudaSuccess) destroy_side(x);
  return e;
}

void destroy_side(SideStream& x) {
  if (x.join) cudaEventDestroy(x.join);
  if (x.fork) cudaEventDestroy(x.fork);
  if (x.st) cudaStreamDestroy(x.st);
  x = SideStream();
}

namespace {

// A second stream for the caller's stream s, marked busy; NULL if there is
// none to be had (another thread is queueing on s's, or all are at work).
SideStream* take_side(fit_handle* h, cudaStream_t s) {
  unsigned long long id = 0;
  if (cudaStreamGetId(s, &id) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(h->side_mu);
  SideStream* found = nullptr;
  for (SideStream& x : h->side)
    if (x.st && x.caller == id) found = &x;
  if (found) {
    if (found->busy) return nullptr;
  } else {
    // (queries and creations that another thread's capture must not mind)
    cudaStreamCaptureMode capture_mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&capture_mode);
    for (SideStream& x : h->side) {
      if (x.busy) continue;
      if (x.st ? cudaStreamQuery(x.st) == cudaSuccess : create_side(x) == cudaSuccess) {
        found = &x;
        break;
      }
      cudaGetLastError();
    }
    cudaThreadExchangeStreamCaptureMode(&capture_mode);
    if (!found) return nullptr;
    found->caller = id;
  }
  found->busy = true;
  return found;
}

}  // namespace

cudaError_t ModeStreams::frontier(Frontier* f, cudaStreamCaptureStatus* status) const {
  const cudaGraphNode_t* nodes = nullptr;
  const cudaGraphEdgeData* edges = nullptr;
  size_t n = 0;
  const cudaError_t e =
      cudaStreamGetCaptureInfo(s_, status, nullptr, nullptr, &nodes, &edges, &n);
  if (e != cudaSuccess || *status != cudaStreamCaptureStatusActive) return e;
  f->nodes.assign(nodes, nodes + n);
  f->edges.assign(edges, edges ? edges + n : edges);
  return e;
}

cudaError_t ModeStreams::depend(Frontier& f, unsigned how) {
  return cudaStreamUpdateCaptureDependencies(s_, f.nodes.data(),
                                             f.edges.empty() ? nullptr : f.edges.data(),
                                             f.nodes.size(), how);
}

int ModeStreams::begin(int nevt, const int64_t* ntrk, const int32_t* mode) {
  bool used[2] = {false, false};
  for (int e = 0; e < nevt; ++e)
    if (ntrk[e] > 0) used[mode[e] == FIT_MODE_Z] = true;
  if (!(used[0] && used[1])) return FIT_OK;
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  if (frontier(&before_, &status) != cudaSuccess) {  // the launches on s_ will say what is wrong
    cudaGetLastError();
    return FIT_OK;
  }
  if (status != cudaStreamCaptureStatusNone) {
    captured_ = status == cudaStreamCaptureStatusActive;
    return FIT_OK;
  }
  side_ = take_side(h_, s_);
  if (!side_) return FIT_OK;
  cudaError_t e = cudaEventRecord(side_->fork, s_);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(side_->st, side_->fork, 0);
  if (e != cudaSuccess)
    return cuda_fail(e, (std::string(who_) + ": fork to the second stream").c_str());
  return FIT_OK;
}

cudaStream_t ModeStreams::of(int m) {
  if (m == FIT_MODE_R) return s_;
  if (side_) return side_->st;
  if (captured_ && !branched_) {
    branched_ = true;
    cudaStreamCaptureStatus status;
    err_ = frontier(&after_r_, &status);
    if (err_ == cudaSuccess) err_ = depend(before_, cudaStreamSetCaptureDependencies);
  }
  return s_;
}

int ModeStreams::end(int rc) {
  cudaError_t e = err_;
  if (side_) {
    e = cudaEventRecord(side_->join, side_->st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s_, side_->join, 0);
  } else if (branched_ && e == cudaSuccess) {
    e = depend(after_r_, cudaStreamAddCaptureDependencies);
  }
  if (e != cudaSuccess && rc == FIT_OK)
    return cuda_fail(e, (std::string(who_) + ": join from the second stream").c_str());
  return rc;
}

ModeStreams::~ModeStreams() {
  if (!side_) return;
  std::lock_guard<std::mutex> lock(h_->side_mu);
  side_->busy = false;
}

int run_fit_streams(fit_handle* h, const FitArgs& a, const RunOptions& o, int nevt,
                    const int64_t* ntrk, const int32_t* mode, const char* who, cudaStream_t s) {
  ModeStreams ms(h, s, who);
  const bool one_launch = !o.seeded && is_small(h, o.call_tracks);
  const int rc = one_launch ? FIT_OK : ms.begin(nevt, ntrk, mode);
  if (rc != FIT_OK) return rc;
  return ms.end(run_fit(h, a, o, nevt, ntrk, mode, who, ms));
}

// Scratch of fit_propagate_update_noalloc, in the library image instead of
// allocated memory: per-event counters [FIT_NOALLOC_MAX_EVENTS][kEventSlots]
// followed by the event offsets [FIT_NOALLOC_MAX_EVENTS + 1] (int64).  Every
// device that loads the library holds it (192 KiB) until the process exits.
constexpr size_t kNoallocCounterWords = (size_t)FIT_NOALLOC_MAX_EVENTS * kEventSlots;
static __device__ __align__(256)
    unsigned long long g_noalloc_scratch[kNoallocCounterWords + FIT_NOALLOC_MAX_EVENTS + 1];

// Device address of g_noalloc_scratch per device.  In host code the array's
// name is only a host-side stand-in, so the address is looked up once per
// device, with that device current, and cached.
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
unsigned long long* g_noalloc_ptr[kMaxDevices] = {};

int noalloc_scratch(int device, unsigned long long** ptr) {
  if (device < 0 || device >= kMaxDevices)
    return fail(FIT_ERR_ARG, "fit_propagate_update_noalloc: device index out of range");
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[device]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "fit_propagate_update_noalloc: cudaGetSymbolAddress");
    g_noalloc_ptr[device] = static_cast<unsigned long long*>(p);
  }
  *ptr = g_noalloc_ptr[device];
  return FIT_OK;
}

}  // namespace fitimpl

using namespace fitimpl;

extern "C" {

const char* fit_last_error(void) { return g_last_error.c_str(); }

int fit_init(fit_handle** out, const fit_config* cfg_r, const fit_config* cfg_z, int device) {
  g_last_error.clear();
  if (!out) return fail(FIT_ERR_ARG, "fit_init: handle pointer is NULL");
  *out = nullptr;
  if (!cfg_r && !cfg_z) return fail(FIT_ERR_ARG, "fit_init: no mode configured");
  int ndev = 0;
  cudaError_t e = cudaGetDeviceCount(&ndev);
  if (e != cudaSuccess) return cuda_fail(e, "fit_init: cudaGetDeviceCount");
  if (device < 0 || device >= ndev) return fail(FIT_ERR_ARG, "fit_init: no such device");
  fit_handle* h = new fit_handle();
  h->device = device;
  int rc = configure_modes(h, cfg_r, cfg_z, "fit_init");
  if (rc != FIT_OK) {
    delete h;
    return rc;
  }
  DeviceGuard g(device);
  e = cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, device);
  if (e != cudaSuccess) {
    delete h;
    return cuda_fail(e, "fit_init: cudaDeviceGetAttribute");
  }
  e = cudaMalloc(&h->d_counters, kCounters * sizeof(unsigned long long));
  if (e != cudaSuccess) {
    delete h;
    return fail(FIT_ERR_NOMEM, std::string("fit_init: cudaMalloc: ") + cudaGetErrorString(e));
  }
  e = cudaMemset(h->d_counters, 0, kCounters * sizeof(unsigned long long));
  if (e == cudaSuccess) e = create_side(h->side[0]);
  if (e != cudaSuccess) {
    cudaFree(h->d_counters);
    delete h;
    return cuda_fail(e, "fit_init: counters, stream and events");
  }
  *out = h;
  return FIT_OK;
}

int fit_propagate_update(fit_handle* h, const fit_tracks_in* in, const fit_tracks_out* out,
                         const fit_hits* hits, int nevt, const int64_t* ntrk, int nlayer,
                         const int32_t* mode, void* stream) {
  g_last_error.clear();
  if (!h) return fail(FIT_ERR_ARG, "fit_propagate_update: NULL argument");
  int64_t total = 0;
  int rc = check_call(h, in, out, hits, nevt, ntrk, nlayer, mode, &total, "fit_propagate_update");
  if (rc != FIT_OK || total == 0) return rc;
  DeviceGuard g(h->device);
  rc = run_fit_streams(h, base_args(in, out, hits, nlayer, h->d_counters),
                       {FIT_LAYOUT_SOA, h->seeded, false, total}, nevt, ntrk, mode,
                       "fit_propagate_update", static_cast<cudaStream_t>(stream));
  if (rc != FIT_OK) return rc;
  h->tracks += (uint64_t)total;
  return FIT_OK;
}

int fit_propagate_update_layout(fit_handle* h, const fit_tracks_in* in, const fit_tracks_out* out,
                                const fit_hits* hits, int nevt, const int64_t* ntrk, int nlayer,
                                const int32_t* mode, int layout, void* stream) {
  static const char* kWho = "fit_propagate_update_layout";
  g_last_error.clear();
  if (!h) return fail(FIT_ERR_ARG, std::string(kWho) + ": NULL argument");
  if (layout == FIT_LAYOUT_SOA)
    return fit_propagate_update(h, in, out, hits, nevt, ntrk, nlayer, mode, stream);
  if (layout != FIT_LAYOUT_AOSOA32) return fail(FIT_ERR_ARG, std::string(kWho) + ": unknown layout");
  int64_t total = 0;
  int rc = check_call(h, in, out, hits, nevt, ntrk, nlayer, mode, &total, kWho);
  if (rc != FIT_OK || total == 0) return rc;
  if ((in->ld | out->ld | hits->ld) & 31)
    return fail(FIT_ERR_ARG, std::string(kWho) + ": AoSoA slots (ld) must be a multiple of 32");
  if (h->seeded) return fail(FIT_ERR_ARG, std::string(kWho) + ": no learned seed in AoSoA");
  DeviceGuard g(h->device);
  rc = run_fit_streams(h, base_args(in, out, hits, nlayer, h->d_counters),
                       {layout, false, false, total}, nevt, ntrk, mode, kWho,
                       static_cast<cudaStream_t>(stream));
  if (rc != FIT_OK) return rc;
  h->tracks += (uint64_t)total;
  return FIT_OK;
}

int fit_propagate_update_noalloc(const fit_config* cfg_r, const fit_config* cfg_z,
                                 const fit_tracks_in* in, const fit_tracks_out* out,
                                 const fit_hits* hits, int nevt, const int64_t* ntrk, int nlayer,
                                 const int32_t* mode, void* stream, fit_status* per_event) {
  static const char* kWho = "fit_propagate_update_noalloc";
  g_last_error.clear();
  if (!cfg_r && !cfg_z) return fail(FIT_ERR_ARG, std::string(kWho) + ": no mode configured");
  if (nevt > FIT_NOALLOC_MAX_EVENTS)
    return fail(FIT_ERR_ARG, std::string(kWho) + ": nevt exceeds FIT_NOALLOC_MAX_EVENTS (" +
                                 std::to_string(FIT_NOALLOC_MAX_EVENTS) +
                                 "); split the events over several calls");
  fit_handle h;  // geometry only; nothing allocated
  int rc = configure_modes(&h, cfg_r, cfg_z, kWho);
  if (rc != FIT_OK) return rc;
  int64_t total = 0;
  rc = check_call(&h, in, out, hits, nevt, ntrk, nlayer, mode, &total, kWho);
  if (rc != FIT_OK) return rc;
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return cuda_fail(e, "fit_propagate_update_noalloc: cudaGetDevice");
  unsigned long long* scratch = nullptr;
  rc = noalloc_scratch(device, &scratch);
  if (rc != FIT_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (nevt > 0) {
    // The counters of this call's events start at zero.
    e = cudaMemsetAsync(scratch, 0, (size_t)nevt * kEventSlots * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return cuda_fail(e, "fit_propagate_update_noalloc: cudaMemsetAsync");
  }
  if (total > 0) {
    const FitArgs args = base_args(in, out, hits, nlayer, scratch);
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return cuda_fail(e, "fit_propagate_update_noalloc: device attribute");
    bool done = false;
    if (is_small(sms, total) && nevt <= kSmallEvents) {
      EventTable<kSmallEvents> ev;
      ev.n = nevt;
      uint32_t t = 0;
      for (int i = 0; i < nevt; ++i) {
        ev.first[i] = t;
        t += (uint32_t)ntrk[i];
      }
      done = launch_small(&h, args, false, nevt, ntrk, mode, [&](const auto& sa, unsigned nblk) {
        fit_small_kernel<0, kSmallEvents><<<nblk, kBlock, 0, s>>>(sa, ev);
      });
    }
    if (!done) {
      // the event offsets, staged from the stack
      int64_t off[FIT_NOALLOC_MAX_EVENTS];
      int64_t t = 0;
      for (int i = 0; i < nevt; ++i) {
        off[i] = t;
        t += ntrk[i];
      }
      int64_t* d_off = reinterpret_cast<int64_t*>(scratch + kNoallocCounterWords);
      e = cudaMemcpyAsync(d_off, off, (size_t)nevt * sizeof(int64_t), cudaMemcpyHostToDevice, s);
      if (e != cudaSuccess) return cuda_fail(e, "fit_propagate_update_noalloc: offset copy");
      rc = launch_runs(&h, args, false, nevt, ntrk, mode, kWho,
                       [=](const FitArgs& a, int m, const PairRuns<kMaxRuns>& r) {
                         if (m == FIT_MODE_Z)
                           fit_fused_kernel_noalloc<FIT_MODE_Z, kMaxRuns>
                               <<<part_blocks<2>(r), kBlock, 0, s>>>(a, r, d_off, nevt);
                         else
                           fit_fused_kernel_noalloc<FIT_MODE_R, kMaxRuns>
                               <<<part_blocks<2>(r), kBlock, 0, s>>>(a, r, d_off, nevt);
                       });
    }
    e = cudaGetLastError();
    if (rc == FIT_OK && e != cudaSuccess)
      rc = cuda_fail(e, "fit_propagate_update_noalloc: launch");
    if (rc != FIT_OK) return rc;
  }
  if (per_event && nevt > 0) {
    static_assert(sizeof(fit_status) == kEventSlots * sizeof(unsigned long long),
                  "fit_status mirrors one row of the per-event counter table");
    e = cudaMemcpyAsync(per_event, scratch, (size_t)nevt * sizeof(fit_status),
                        cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return cuda_fail(e, "fit_propagate_update_noalloc: counter copy");
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "fit_propagate_update_noalloc: cudaStreamSynchronize");
    for (int i = 0; i < nevt; ++i) per_event[i].tracks = (uint64_t)ntrk[i];
  }
  return FIT_OK;
}

int fit_sync(fit_handle* h, void* stream, double timeout_s, fit_status* st) {
  g_last_error.clear();
  if (!h) return fail(FIT_ERR_ARG, "fit_sync: handle is NULL");
  DeviceGuard g(h->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (timeout_s > 0) {
    const auto deadline = std::chrono::steady_clock::now() + std::chrono::duration<double>(timeout_s);
    for (;;) {
      cudaError_t q = cudaStreamQuery(s);
      if (q == cudaSuccess) break;
      if (q != cudaErrorNotReady) return cuda_fail(q, "fit_sync: cudaStreamQuery");
      if (std::chrono::steady_clock::now() > deadline)
        return fail(FIT_ERR_TIMEOUT, "fit_sync: timed out waiting for the stream");
      std::this_thread::sleep_for(std::chrono::microseconds(50));
    }
  }
  unsigned long long c[kCounters] = {0, 0, 0, 0, 0};
  cudaError_t e = cudaMemcpyAsync(c, h->d_counters, sizeof(c), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return cuda_fail(e, "fit_sync: counter copy");
  e = cudaMemsetAsync(h->d_counters, 0, sizeof(c), s);
  if (e != cudaSuccess) return cuda_fail(e, "fit_sync: counter reset");
  e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "fit_sync: cudaStreamSynchronize");
  if (st) {
    st->tracks = h->tracks;
    st->no_intersection = c[0];
    st->not_converged = c[1];
    st->nonfinite = c[2];
    st->charge_flip = c[3];
    st->iterations = c[4];
  }
  h->tracks = 0;
  return FIT_OK;
}

void fit_destroy(fit_handle* h) {
  if (!h) return;
  {
    DeviceGuard g(h->device);
    if (h->d_counters || h->d_mlp || h->host_stage) cudaDeviceSynchronize();
    if (h->d_counters) cudaFree(h->d_counters);
    if (h->d_mlp) cudaFree(h->d_mlp);
    for (SideStream& x : h->side) destroy_side(x);
    destroy_host_stage(h);
  }
  delete h;
}

}  // extern "C"
