// The FP64 variant of the fused fit: the per-track math of fit_fused_kernel
// (track_math.cuh) instantiated on double, one track per thread, on double
// structure-of-arrays buffers.  The paper's test codes ran in double by
// default (Sec. 5, the FP32 runs are the exception); this variant measures
// what GB300's reduced FP64 rate costs on the same path.
#include <cuda_runtime.h>

#include <cstdint>
#include <string>

#include "fit.h"
#include "fused.cuh"
#include "internal.h"

using namespace fitimpl;

namespace {

// The FP64 pipe is the bound, so an SM that runs one block more than the
// average sets the time: 375 blocks of 128 (48000 tracks) are 2.5 an SM and
// take three, 750 of 64 are 4.9 and take five.
constexpr int kBlock64 = 64;

struct Args64 {
  const double* par_in;
  const double* cov_in;
  const int32_t* q_in;
  int64_t ld_in;
  double* par_out;
  double* cov_out;
  int32_t* q_out;
  double* chi2;
  double* chi2_layer;
  uint8_t* status;
  int64_t ld_out;
  const double* hpos;
  const double* hcov;
  int64_t ld_hit;
  int64_t t0;  // base of the run table
  int nlayer;
  double kB;  // kA * B in double
  unsigned long long* counters;
  Geo geo;
};

// One track per thread over all layers; status bits, per-layer chi2 and
// counters as fit_fused_kernel, and the covariance in the same loop form
// (fused.cuh, enter_loop_form): p2z with its zero z row, p2r in the
// cylinder's local coordinates.
template <int MODE>
__global__ void __launch_bounds__(kBlock64)
    fit_f64_kernel(const __grid_constant__ Args64 a, const __grid_constant__ TrackRuns r) {
  const unsigned i = blockIdx.x * kBlock64 + threadIdx.x;
  if (i >= r.n) return;
  const int64_t t = a.t0 + run_element(r, i, 1);
  double p[6], c[21], cl[15], bc = 0.0, bs = 0.0;
#pragma unroll
  for (int k = 0; k < 6; ++k) fitk::ld(p[k], a.par_in + k * a.ld_in + t);
#pragma unroll
  for (int k = 0; k < 21; ++k) fitk::ld(c[k], a.cov_in + k * a.ld_in + t);
  double qf = (double)__ldcs(a.q_in + t);
  double chi2 = 0.0;
  fitk::Trig<double> g = fitk::trig_of(p);
  {
    const double kappa = qf * -a.kB * p[3];
    if (MODE == FIT_MODE_Z) {
      fitk::enter_plane(c, g, kappa);
    } else {
      fitk::enter_line(c, g, kappa, cl);
      bc = g.cphi;
      bs = g.sphi;
    }
  }
  bool moved = false;  // some propagation was applied
  unsigned st = 0u, iters[1] = {0u};
  const Geo& geo = a.geo;
  const int64_t ldh = a.ld_hit;
  for (int l = 0; l < a.nlayer; ++l) {
    double m[3], v[6];
#pragma unroll
    for (int k = 0; k < 3; ++k) fitk::ld(m[k], a.hpos + (3 * l + k) * ldh + t);
#pragma unroll
    for (int k = 0; k < 6; ++k) fitk::ld(v[k], a.hcov + (6 * l + k) * ldh + t);
    const float sf = geo.surf.s[l];
    const double dkdw = qf * -a.kB;
    bool nc = false, failed;
    double lag = 0.0;
    if (MODE == FIT_MODE_Z)
      failed = fitk::prop_z<true>(p, c, g, dkdw, sf);
    else
      failed = fitk::prop_r_local(p, cl, bc, bs, g, dkdw, sf, geo.max_iter, geo.tol * sf,
                                  geo.line_start, iters, nc, lag);
    if (failed) {
      st |= FIT_ST_NO_INTERSECTION;
      if (a.chi2_layer)
        for (int r = l; r < a.nlayer; ++r) a.chi2_layer[(int64_t)r * a.ld_out + t] = 0.0;
      break;
    }
    moved = true;
    const double phi_pred = p[4], th_pred = p[5];
    double x2;
    bool flip;
    if (MODE == FIT_MODE_Z) {
      x2 = fitk::update_z<true>(p, c, m, v);
      flip = fitk::normalise(p, c, qf, g, phi_pred, th_pred);
    } else {
      x2 = fitk::update_r_local(p, cl, bc, bs, m, v);
      flip = fitk::normalise(p, cl, qf, g, phi_pred, th_pred, lag);
    }
    const bool alive = fitk::finite_(x2);
    if (nc) st |= FIT_ST_NOT_CONVERGED;
    if (flip) st |= FIT_ST_CHARGE_FLIP;
    if (!alive) st |= FIT_ST_NONFINITE;
    x2 = alive ? x2 : 0.0;
    chi2 += x2;
    if (a.chi2_layer) a.chi2_layer[(int64_t)l * a.ld_out + t] = x2;
    if (!alive) {
      if (a.chi2_layer)
        for (int r = l + 1; r < a.nlayer; ++r) a.chi2_layer[(int64_t)r * a.ld_out + t] = 0.0;
      break;
    }
  }
  if (!moved) {  // nothing applied: the input covariance
#pragma unroll
    for (int k = 0; k < 21; ++k) fitk::ld(c[k], a.cov_in + k * a.ld_in + t);
  } else if (MODE == FIT_MODE_R) {
    fitk::to_global_r(cl, bc, bs, c);
  }
  bool fin = isfinite(chi2);
#pragma unroll
  for (int k = 0; k < 6; ++k) fin = fin && isfinite(p[k]);
#pragma unroll
  for (int k = 0; k < 21; ++k) fin = fin && isfinite(c[k]);
  if (!fin) st |= FIT_ST_NONFINITE;
#pragma unroll
  for (int k = 0; k < 6; ++k) a.par_out[k * a.ld_out + t] = p[k];
#pragma unroll
  for (int k = 0; k < 21; ++k) a.cov_out[k * a.ld_out + t] = c[k];
  a.chi2[t] = chi2;
  a.q_out[t] = (int32_t)qf;
  if (a.status) a.status[t] = (uint8_t)st;
  if (st) count_status(st, a.counters);
  if (MODE == FIT_MODE_R) count_iterations(iters[0], &a.counters[4]);
}

bool aligned8(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 7u) == 0; }

}  // namespace

extern "C" int fit_propagate_update_f64(fit_handle* h, const fit_tracks_in_f64* in,
                                        const fit_tracks_out_f64* out, const fit_hits_f64* hits,
                                        int nevt, const int64_t* ntrk, int nlayer,
                                        const int32_t* mode, void* stream) {
  static const std::string w = "fit_propagate_update_f64";
  g_last_error.clear();
  if (!h || !in || !out || !hits) return fail(FIT_ERR_ARG, w + ": NULL argument");
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
  if (total == 0) return FIT_OK;
  if (!in->par || !in->cov || !in->q || !out->par || !out->cov || !out->q || !out->chi2 ||
      !hits->pos || !hits->cov)
    return fail(FIT_ERR_ARG, w + ": NULL data pointer");
  const void* ptrs[] = {in->par, in->cov, out->par, out->cov, out->chi2, hits->pos, hits->cov};
  for (const void* p : ptrs)
    if (!aligned8(p)) return fail(FIT_ERR_ARG, w + ": pointer not 8-byte aligned");
  if (in->ld < total || out->ld < total || hits->ld < total)
    return fail(FIT_ERR_ARG, w + ": ld smaller than the number of tracks");
  DeviceGuard guard(h->device);
  Args64 a{};
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
  a.counters = h->d_counters;
  // Side by side the two modes' blocks spread unevenly over the FP64 pipes, and
  // a call of many waves is slower for it (96000 tracks 1354 against 1212 us);
  // one of a single wave takes the longer mode's time instead of the sum (608
  // to 9728 tracks 243 us against 411 to 426).  Taken where every block has an
  // SM to itself; up to twice as many tracks still gain (19456 260 against
  // 427, with a tenth of them p2r 344 against 444).
  ModeStreams ms(h, static_cast<cudaStream_t>(stream), w.c_str());
  int rc = total <= (int64_t)kBlock64 * h->sms ? ms.begin(nevt, ntrk, mode) : FIT_OK;
  if (rc != FIT_OK) return rc;
  for (int m : {FIT_MODE_R, FIT_MODE_Z}) {  // one launch per mode
    const cudaStream_t s = ms.of(m);
    a.geo = h->geo[m];
    a.kB = 0.00299792458 * (double)h->B[m];
    rc = launch_track_runs(nevt, ntrk, mode, m, w.c_str(), [&](int64_t t0, const TrackRuns& r) {
      a.t0 = t0;
      const unsigned nblk = (r.n + kBlock64 - 1) / kBlock64;
      if (m == FIT_MODE_Z)
        fit_f64_kernel<FIT_MODE_Z><<<nblk, kBlock64, 0, s>>>(a, r);
      else
        fit_f64_kernel<FIT_MODE_R><<<nblk, kBlock64, 0, s>>>(a, r);
    });
    if (rc != FIT_OK) break;
  }
  rc = ms.end(rc);
  if (rc != FIT_OK) return rc;
  h->tracks += (uint64_t)total;
  return FIT_OK;
}
