// Track finding: on each layer the track is propagated and every candidate
// hit is tried against the prediction; the candidate with the smallest chi2
// strictly below the gate (the lowest index among equal chi2) updates the
// track, or none does and the track keeps its prediction.  The hit choice of
// mkFit's pattern recognition that the paper's test codes leave out (they
// take the one hit given, Sec. 3); the per-track math is the fused fit's
// (track_math.cuh), in FP32 or FP64, one track per thread.
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <type_traits>

#include "fit.h"
#include "fused.cuh"
#include "internal.h"

using namespace fitimpl;

namespace {

constexpr int kMaxCand = 16;

template <class T>
struct FindArgs {
  const T* par_in;
  const T* cov_in;
  const int32_t* q_in;
  int64_t ld_in;
  T* par_out;
  T* cov_out;
  int32_t* q_out;
  T* chi2;
  T* chi2_layer;
  uint8_t* status;
  int64_t ld_out;
  const T* cpos;  // [nlayer][ncand][3][ld_cand]
  const T* ccov;  // [nlayer][ncand][6][ld_cand]
  int ncand;
  int64_t ld_cand;
  int8_t* chosen;  // [nlayer][ld_out]
  T gate;
  int64_t t0;  // base of the run table
  int nlayer;
  T kB;
  unsigned long long* counters;
  Geo geo;
};

// Candidates in registers: slot k mod S holds candidate k of the layer, and is
// refilled (with candidate k + S, or with the next layer's candidate k) as
// soon as candidate k has been tried, so that the loads' latency passes
// behind the other candidates, the update and the next propagation, and the
// update takes its candidate from registers.  Loaded one at a time and the
// chosen one again, the p2r kernel waited on loads 8.2 cycles an instruction
// (now 0.9): 240k tracks, 4 candidates, 20 layers 217 -> 175 us, and both
// modes of that size 383 -> 246 us with p2z on the second stream.  Four
// slots (two with 6 and 7 blocks an SM for p2r and p2z 265 us, three with 5
// and 6 288).  In double, bound by the FP64 pipe, one slot is enough.
//
// Five blocks of 128 an SM in float (96 registers; p2r spills 72 bytes in
// order and 56 with addresses formed anew, p2z none).  Four (no spills) are
// 3 to 9 % faster up to 200000 tracks of p2r -- 48000 with 4 candidates 47.5
// us against 50.7, with 9 89.8 against 94.5 -- and up to 10 % slower beyond:
// 480000 with 4 candidates 311 against 297, with 9 636 against 579, both modes
// with 4 256 against 250.  The long calls decide.
template <class T>
constexpr int kSlots = sizeof(T) == 4 ? 4 : 1;
// In order: the slots are refilled in the order the candidates lie in memory,
// which holds for up to S candidates and for multiples of S.  Then two running
// pointers step through the rows; otherwise every candidate's address is
// formed anew (the usual 4 candidates: 246 against 261 us).
bool in_order(int ncand, int slots) { return ncand <= slots || ncand % slots == 0; }

template <int MODE, class T, bool SEQ>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 8 ? 1 : 5)
    fit_find_kernel(const __grid_constant__ FindArgs<T> a, const __grid_constant__ TrackRuns r) {
  const unsigned i = blockIdx.x * kBlock + threadIdx.x;
  if (i >= r.n) return;
  const int64_t t = a.t0 + run_element(r, i, 1);
  // The covariance in the fused fit's loop form (fused.cuh, enter_loop_form):
  // p2z c with a zero z row, p2r the local form cl with the null direction
  // (bc, bs).
  T p[6], c[21], cl[15], bc, bs;
#pragma unroll
  for (int k = 0; k < 6; ++k) fitk::ld(p[k], a.par_in + k * a.ld_in + t);
#pragma unroll
  for (int k = 0; k < 21; ++k) fitk::ld(c[k], a.cov_in + k * a.ld_in + t);
  T qf = (T)__ldcs(a.q_in + t);
  T chi2 = T(0.f);
  fitk::Trig<T> g = fitk::trig_of(p);
  {
    const T kappa = qf * -a.kB * p[3];
    if (MODE == FIT_MODE_Z) {
      fitk::enter_plane(c, g, kappa);
    } else {
      fitk::enter_line(c, g, kappa, cl);
      bc = g.cphi;
      bs = g.sphi;
    }
  }
  unsigned st = 0u, iters[1] = {0u};
  const Geo& geo = a.geo;
  const int64_t ldc = a.ld_cand;
  constexpr int S = kSlots<T>;
  T sm[S][3], sv[S][6];
  const T* qp = a.cpos + t;
  const T* qc = a.ccov + t;
  // candidate k of layer l into slot j
  auto fill = [&](int j, int l, int k) {
    if constexpr (!SEQ) {
      const int64_t row = (int64_t)l * a.ncand + k;
      qp = a.cpos + 3 * row * ldc + t;
      qc = a.ccov + 6 * row * ldc + t;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i, qp += ldc) fitk::ld(sm[j][i], qp);
#pragma unroll
    for (int i = 0; i < 6; ++i, qc += ldc) fitk::ld(sv[j][i], qc);
  };
#pragma unroll
  for (int j = 0; j < S; ++j)
    if (j < a.ncand && a.nlayer > 0) fill(j, 0, j);
  // The layer loop runs the p2r crossing start in its series form only
  // (Start::kFast).  A surface where that form does not apply ends the inner
  // loop; the outer one then propagates to it from crossing_exact's start and
  // resumes the inner loop at its candidates.  Kept out of the inner loop,
  // the exact form costs the loop nothing (inside it, 20 %).
  int l = 0;
  bool propagated = false;  // layer l's propagation is done
  T lag = T(0.f);           // p2r: how far (g.cphi, g.sphi) trails p[4] (prop_r_local)
  for (;;) {
    bool rerun = false;
    for (; l < a.nlayer; ++l) {
      const float sf = geo.surf.s[l];
      const T dkdw = qf * -a.kB;
      bool nc = false, failed = false;
      if (propagated)
        propagated = false;
      else if (MODE == FIT_MODE_Z)
        failed = fitk::prop_z<true>(p, c, g, dkdw, sf);
      else
        failed = fitk::prop_r_local<T, fitk::Start::kFast>(p, cl, bc, bs, g, dkdw, sf,
                                                           geo.max_iter, geo.tol * sf,
                                                           geo.line_start, iters, nc, lag);
      if (failed) {
        if (MODE == FIT_MODE_R && !geo.line_start)
          rerun = true;
        else
          st |= FIT_ST_NO_INTERSECTION;
        break;
      }
      if (nc) st |= FIT_ST_NOT_CONVERGED;
      int best = -1;
      T best_chi2 = a.gate;
      T m[3], v[6];  // the best candidate so far
      for (int k0 = 0; k0 < a.ncand; k0 += S) {
#pragma unroll
        for (int j = 0; j < S; ++j) {
          const int k = k0 + j;
          if (k >= a.ncand) break;
          const T x = (MODE == FIT_MODE_Z) ? fitk::chi2_z(p, c, sm[j], sv[j])
                                           : fitk::chi2_r_local(p, cl, bc, bs, sm[j], sv[j]);
          if (x < best_chi2) {
            best = k;
            best_chi2 = x;
#pragma unroll
            for (int i = 0; i < 3; ++i) m[i] = sm[j][i];
#pragma unroll
            for (int i = 0; i < 6; ++i) v[i] = sv[j][i];
          }
          if (k + S < a.ncand)
            fill(j, l, k + S);
          else if (l + 1 < a.nlayer)
            fill(j, l + 1, j);
        }
      }
      a.chosen[(int64_t)l * a.ld_out + t] = (int8_t)best;
      T x2 = T(0.f);
      if (best >= 0) {
        const T phi_pred = p[4], th_pred = p[5];
        bool flip;
        if (MODE == FIT_MODE_Z) {
          x2 = fitk::update_z<true>(p, c, m, v);
          flip = fitk::normalise(p, c, qf, g, phi_pred, th_pred);
        } else {
          x2 = fitk::update_r_local(p, cl, bc, bs, m, v);
          flip = fitk::normalise(p, cl, qf, g, phi_pred, th_pred, lag);
        }
        if (flip) st |= FIT_ST_CHARGE_FLIP;
        if (!fitk::finite_(x2)) {
          st |= FIT_ST_NONFINITE;
          x2 = T(0.f);
          if (a.chi2_layer) a.chi2_layer[(int64_t)l * a.ld_out + t] = x2;
          ++l;
          break;
        }
      } else if (MODE == FIT_MODE_R) {
        fitk::turn_by(g.cphi, g.sphi, lag);  // no update: the propagation's own turn
      }
      chi2 += x2;
      if (a.chi2_layer) a.chi2_layer[(int64_t)l * a.ld_out + t] = x2;
    }
    if (!rerun) break;
    const float sf = geo.surf.s[l];
    const T dkdw = qf * -a.kB;
    const T h0 = fitk::crossing_exact<T>(p[0], p[1], g.cphi, g.sphi, dkdw * p[3], T(sf));
    bool nc = false;
    if (fitk::prop_r_local<T, fitk::Start::kGiven>(p, cl, bc, bs, g, dkdw, sf, geo.max_iter,
                                                   geo.tol * sf, false, iters, nc, lag, h0)) {
      st |= FIT_ST_NO_INTERSECTION;
      break;
    }
    if (nc) st |= FIT_ST_NOT_CONVERGED;
    propagated = true;
  }
  for (int k = l; k < a.nlayer; ++k) {  // layers not reached
    a.chosen[(int64_t)k * a.ld_out + t] = -1;
    if (a.chi2_layer) a.chi2_layer[(int64_t)k * a.ld_out + t] = T(0.f);
  }
  if (l == 0) {  // nothing applied: the input covariance
#pragma unroll
    for (int k = 0; k < 21; ++k) fitk::ld(c[k], a.cov_in + k * a.ld_in + t);
  } else if (MODE == FIT_MODE_R) {
    fitk::to_global_r(cl, bc, bs, c);
  }
  bool fin = fitk::finite_(chi2);
#pragma unroll
  for (int k = 0; k < 6; ++k) fin = fin && fitk::finite_(p[k]);
#pragma unroll
  for (int k = 0; k < 21; ++k) fin = fin && fitk::finite_(c[k]);
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

bool aligned(const void* p, unsigned a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

template <class T, class In, class Out, class Cand>
int find_tracks(fit_handle* h, const In* in, const Out* out, const Cand* cand, double gate,
                int8_t* chosen, int nevt, const int64_t* ntrk, int nlayer, const int32_t* mode,
                void* stream, const std::string& w) {
  g_last_error.clear();
  if (!h || !in || !out || !cand || !chosen) return fail(FIT_ERR_ARG, w + ": NULL argument");
  if (nevt < 0) return fail(FIT_ERR_ARG, w + ": nevt < 0");
  if (nevt > 0 && (!ntrk || !mode)) return fail(FIT_ERR_ARG, w + ": ntrk or mode is NULL");
  if (cand->ncand < 1 || cand->ncand > kMaxCand)
    return fail(FIT_ERR_ARG, w + ": ncand out of [1, 16]");
  if (!(gate > 0.0)) return fail(FIT_ERR_ARG, w + ": chi2_gate must be > 0");
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
      !cand->pos || !cand->cov)
    return fail(FIT_ERR_ARG, w + ": NULL data pointer");
  const void* ptrs[] = {in->par, in->cov, out->par, out->cov, out->chi2, cand->pos, cand->cov};
  for (const void* p : ptrs)
    if (!aligned(p, sizeof(T))) return fail(FIT_ERR_ARG, w + ": misaligned pointer");
  if (in->ld < total || out->ld < total || cand->ld < total)
    return fail(FIT_ERR_ARG, w + ": ld smaller than the number of tracks");
  DeviceGuard guard(h->device);
  FindArgs<T> a{};
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
  a.cpos = cand->pos;
  a.ccov = cand->cov;
  a.ncand = cand->ncand;
  a.ld_cand = cand->ld;
  a.chosen = chosen;
  a.gate = (T)gate;
  a.nlayer = nlayer;
  a.counters = h->d_counters;
  ModeStreams ms(h, static_cast<cudaStream_t>(stream), w.c_str());
  int rc = ms.begin(nevt, ntrk, mode);
  if (rc != FIT_OK) return rc;
  for (int m : {FIT_MODE_R, FIT_MODE_Z}) {  // one launch per mode
    const cudaStream_t s = ms.of(m);
    a.geo = h->geo[m];
    a.kB = sizeof(T) == 8 ? (T)(0.00299792458 * (double)h->B[m]) : (T)h->geo[m].kB;
    rc = launch_track_runs(nevt, ntrk, mode, m, w.c_str(), [&](int64_t t0, const TrackRuns& r) {
      a.t0 = t0;
      const unsigned nblk = (r.n + kBlock - 1) / kBlock;
      auto launch = [&](auto seq) {
        constexpr bool SEQ = decltype(seq)::value;
        if (m == FIT_MODE_Z)
          fit_find_kernel<FIT_MODE_Z, T, SEQ><<<nblk, kBlock, 0, s>>>(a, r);
        else
          fit_find_kernel<FIT_MODE_R, T, SEQ><<<nblk, kBlock, 0, s>>>(a, r);
      };
      if constexpr (kSlots<T> > 1) {
        if (!in_order(a.ncand, kSlots<T>)) return launch(std::false_type());
      }
      launch(std::true_type());
    });
    if (rc != FIT_OK) break;
  }
  rc = ms.end(rc);
  if (rc != FIT_OK) return rc;
  h->tracks += (uint64_t)total;
  return FIT_OK;
}

}  // namespace

extern "C" int fit_find_tracks(fit_handle* h, const fit_tracks_in* in, const fit_tracks_out* out,
                               const fit_candidates* cand, float chi2_gate, int8_t* chosen,
                               int nevt, const int64_t* ntrk, int nlayer, const int32_t* mode,
                               void* stream) {
  return find_tracks<float>(h, in, out, cand, chi2_gate, chosen, nevt, ntrk, nlayer, mode, stream,
                            "fit_find_tracks");
}

extern "C" int fit_find_tracks_f64(fit_handle* h, const fit_tracks_in_f64* in,
                                   const fit_tracks_out_f64* out, const fit_candidates_f64* cand,
                                   double chi2_gate, int8_t* chosen, int nevt, const int64_t* ntrk,
                                   int nlayer, const int32_t* mode, void* stream) {
  return find_tracks<double>(h, in, out, cand, chi2_gate, chosen, nevt, ntrk, nlayer, mode, stream,
                             "fit_find_tracks_f64");
}
