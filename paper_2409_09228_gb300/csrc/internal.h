// Internal declarations shared by the libfit translation units (not part of
// the C ABI).  Host-side helpers and the kernel argument blocks.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>
#include <string>
#include <vector>

#include "fit.h"

namespace fitimpl {

// Error reporting: the message of the last failure on the calling thread.
extern thread_local std::string g_last_error;
int fail(int code, const std::string& msg);
int cuda_fail(cudaError_t e, const char* what);

constexpr int kBlock = 128;
constexpr int kCounters = 5;  // no_intersection, not_converged, nonfinite, charge_flip,
                               // p2r path-length iterations

struct Surfaces {
  float s[FIT_MAX_LAYERS];
};

// Geometry and numerics of one mode.
struct Geo {
  float kB;  // kA * B
  int max_iter;
  float tol;
  int line_start;  // p2r: start the path-length iteration at the straight-line step
  Surfaces surf;
};

struct FitArgs {
  const float* par_in;
  const float* cov_in;
  const int32_t* q_in;
  int64_t ld_in;
  float* par_out;
  float* cov_out;
  int32_t* q_out;
  float* chi2;
  float* chi2_layer;
  uint8_t* status;
  int64_t ld_out;
  const float* hpos;
  const float* hcov;
  int64_t ld_hit;
  int64_t t0;  // the track that the launch's run table counts from
  int nlayer;
  unsigned long long* counters;
  Geo geo;
};

// The tracks of one launch: runs of same-mode events, which other events'
// tracks separate, as one list of elements (tracks, or pairs of tracks).
// Element i lies in the run r with the largest before[r] <= i, at track
// first[r] + stride * (i - before[r]) counted from the launch's FitArgs::t0.
// The tables travel as kernel parameters: no allocation, no copy to wait for,
// nothing to keep alive, and a captured launch holds its own.
template <int K>
struct Runs {
  int nrun;
  uint32_t n;  // elements
  uint32_t first[K];
  uint32_t before[K];
};

// Runs as pairs of tracks (2 k, 2 k + 1) for the packed kernels, and the
// tracks that a run's odd edges leave without a partner.
template <int K>
struct PairRuns {
  Runs<K> pairs;
  uint32_t nlone;
  uint32_t lone[2 * K];
};

// Capacities compiled: the usual call has one run per mode; a call of uneven
// mixed events has hundreds.  kMaxRuns pair runs take 16 KiB of parameters.
constexpr int kMaxRuns = 1024;
constexpr int kSmallRuns = 256;  // of each mode, in a small call's one launch

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

class DeviceGuard {
 public:
  explicit DeviceGuard(int dev) : dev_(dev) {
    cudaGetDevice(&prev_);
    if (prev_ != dev_) cudaSetDevice(dev_);
  }
  ~DeviceGuard() {
    if (prev_ != dev_) cudaSetDevice(prev_);
  }

 private:
  int dev_, prev_ = 0;
};


// A second stream of a handle (ModeStreams).
struct SideStream {
  cudaStream_t st = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
  unsigned long long caller = 0;  // id of the stream that it served last
  bool busy = false;              // a call is queueing on it
};
constexpr int kSideStreams = 8;
cudaError_t create_side(SideStream& x);
void destroy_side(SideStream& x);

}  // namespace fitimpl


struct fit_handle {
  int device = 0;
  int sms = 0;  // streaming multiprocessors of the device
  bool has[2] = {false, false};
  int nlayer[2] = {0, 0};
  fitimpl::Geo geo[2];
  unsigned long long* d_counters = nullptr;  // [kCounters]
  uint64_t tracks = 0;
  void* d_mlp = nullptr;  // learned-seed weights (fit_mlp_attach), device
  bool seeded = false;    // p2r seeds from d_mlp
  void* host_stage = nullptr;  // staging of fit_propagate_update_host (host.cu)
  float B[2] = {0.f, 0.f};     // field of each mode's configuration
  fitimpl::SideStream side[fitimpl::kSideStreams];  // the first from fit_init, others when needed
  std::mutex side_mu;  // guards the entries' taking and giving back
};


namespace fitimpl {

// Argument checks shared by the entry points that run the fused kernel.
int check_call(const fit_handle* h, const fit_tracks_in* in, const fit_tracks_out* out,
               const fit_hits* hits, int nevt, const int64_t* ntrk, int nlayer,
               const int32_t* mode, int64_t* total_out, const char* who);
FitArgs base_args(const fit_tracks_in* in, const fit_tracks_out* out, const fit_hits* hits,
                  int nlayer, unsigned long long* counters);

// The p2r events of a fit seeded by the learned path length (mlp.cu), one
// track per thread.
int launch_seeded_fit(const fit_handle* h, const FitArgs& a, int nevt, const int64_t* ntrk,
                      const int32_t* mode, const char* who, cudaStream_t s);

// The kernels with one track per thread: the tracks of mode m's events as
// run tables of up to kTrackRuns runs (1 KiB of parameters, which costs a
// launch nothing measurable), launch(base, r) for each; returns FIT_OK or the
// first launch's error.  A stream of more runs takes several launches, each
// with a last wave of its own: 600 mixed events, 40000 tracks, finder 130,
// adjoint 300, FP64 894 us; with tables of 1024 runs 74, 173 and 592, and a
// call of one run unchanged (171 us).
constexpr int kTrackRuns = 128;
using TrackRuns = Runs<kTrackRuns>;

template <class Launch>
int launch_track_runs(int nevt, const int64_t* ntrk, const int32_t* mode, int m, const char* who,
                      Launch launch) {
  TrackRuns r;
  r.nrun = 0, r.n = 0;
  int64_t base = 0, t = 0;
  auto flush = [&]() {
    if (!r.n) return FIT_OK;
    launch(base, r);
    r.nrun = 0, r.n = 0;
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? FIT_OK : cuda_fail(e, (std::string(who) + ": launch").c_str());
  };
  constexpr int64_t kSpan = int64_t(1) << 31;
  for (int e = 0; e < nevt; ++e) {
    int64_t t1 = t + ntrk[e];
    if (mode[e] == m) {
      while (e + 1 < nevt && mode[e + 1] == m) t1 += ntrk[++e];
      while (t < t1) {
        if (!r.nrun) base = t;
        const int64_t end = base + kSpan < t1 ? base + kSpan : t1;
        if (r.nrun == kTrackRuns || end <= t) {
          const int rc = flush();
          if (rc != FIT_OK) return rc;
          continue;
        }
        r.first[r.nrun] = (uint32_t)(t - base);
        r.before[r.nrun++] = r.n;
        r.n += (uint32_t)(end - t);
        t = end;
      }
    }
    t = t1;
  }
  return flush();
}

// How run_fit takes a call's events.
struct RunOptions {
  int layout = FIT_LAYOUT_SOA;
  bool seeded = false;      // the p2r events start from the handle's learned seed
  bool by_event = false;    // pairs never cross an event (else: a run of same-mode events)
  int64_t call_tracks = 0;  // tracks of the whole call, which may be cut into chunks
};

// The two modes' events of a call are independent: with both present, the
// p2z launches go to a second stream, so that they overlap the p2r launches
// (their blocks fill the SMs a launch's last wave leaves idle).  begin() forks
// it from the caller's stream s, of(m) is the stream for a launch of mode m
// (the p2r launches first), and end(rc) joins it back (even after a failed
// launch, so that s still follows everything that was queued) and returns rc
// or the first error of its own.  Without begin() every launch goes to s.
//
// Calls on different streams must not wait for one another, so each has a
// second stream of its own: the one that served the same caller's stream
// before, or one that is idle, or a new one, or, with all kSideStreams at
// work, none -- the launches then follow one another on s.  Under capture no
// second stream is used (it would belong to the capture until that ends, and
// refuse every other call): the p2z launches become a branch of the graph by
// setting the capture's dependencies back to those of begin().
class ModeStreams {
 public:
  ModeStreams(fit_handle* h, cudaStream_t s, const char* who) : h_(h), s_(s), who_(who) {}
  ~ModeStreams();
  ModeStreams(const ModeStreams&) = delete;
  ModeStreams& operator=(const ModeStreams&) = delete;
  int begin(int nevt, const int64_t* ntrk, const int32_t* mode);
  cudaStream_t of(int m);
  int end(int rc);

 private:
  // What the next captured operation depends on.
  struct Frontier {
    std::vector<cudaGraphNode_t> nodes;
    std::vector<cudaGraphEdgeData> edges;  // empty, or one per node
  };
  cudaError_t frontier(Frontier* f, cudaStreamCaptureStatus* status) const;
  cudaError_t depend(Frontier& f, unsigned how);

  fit_handle* h_;
  cudaStream_t s_;
  const char* who_;
  SideStream* side_ = nullptr;
  bool captured_ = false, branched_ = false;
  Frontier before_, after_r_;
  cudaError_t err_ = cudaSuccess;
};

// The fused fit of events [0, nevt) (fit.cu): the p2r events in one launch
// (kMaxRuns runs each), the p2z events in one, on ms's streams; a small call
// in one launch.
int run_fit(const fit_handle* h, const FitArgs& a, const RunOptions& o, int nevt,
            const int64_t* ntrk, const int32_t* mode, const char* who, ModeStreams& ms);

// run_fit with a second stream for p2z where both modes are present.
int run_fit_streams(fit_handle* h, const FitArgs& a, const RunOptions& o, int nevt,
                    const int64_t* ntrk, const int32_t* mode, const char* who, cudaStream_t s);

// Frees the staging of fit_propagate_update_host (host.cu).
void destroy_host_stage(fit_handle* h);

}  // namespace fitimpl
