"""A call's events gathered into one launch per mode (the run tables): more
runs of same-mode events than one table holds, runs that begin and end at odd
tracks, runs of a single track, empty events."""
import numpy as np
import pytest

import oracle
import parity
from paper_2409_09228_gb300 import fit, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("needs a CUDA device", allow_module_level=True)

import gpu_util  # noqa: E402

NLAYER = 20


def _events(nevt, seed=61):
    """nevt events, modes alternating, 0..5 tracks each (the first one odd)."""
    nt = np.array([1, 2, 3, 1, 5, 0, 4, 1, 1, 2, 0])[np.arange(nevt) % 11]
    return inputs.generate_events(nt, np.arange(nevt) % 2, seed=seed, nlayer=NLAYER)


def _device(ev, ld, dtype=None):
    d = [gpu_util.to_dev(a, ld) for a in (ev.par0, ev.cov0, ev.q, ev.hpos, ev.hcov)]
    return d if dtype is None else [a.to(dtype) if k != 2 else a for k, a in enumerate(d)]


def _fitter(ev):
    return fit.Fitter(fit.Geometry(ev.B, ev.surf[0]), fit.Geometry(ev.B, ev.surf[1]))


def _of_mode(ev, m):
    return np.nonzero(np.repeat(ev.mode, ev.ntrk) == m)[0]


def _check(ev, got, label):
    for m in (0, 1):
        idx = _of_mode(ev, m)
        if not len(idx):
            continue
        ts = inputs.TrackSet(m, ev.B, ev.surf[m], *(np.ascontiguousarray(a[..., idx]) for a in
                                                    (ev.par0, ev.cov0, ev.q, ev.hpos, ev.hcov)))
        parity.check({k: v[..., idx] for k, v in got.items()}, oracle.fit_set(ts), f"{label} mode {m}")


# 7 runs: every mode in one small table; 2303: two full tables of 1024 a mode
@pytest.mark.parametrize("nevt", [1, 7, 2303])
@pytest.mark.parametrize("entry", ["fit", "aosoa", "noalloc", "plan"])
def test_pair_kernels_many_runs(entry, nevt):
    ev = _events(nevt)
    ld = (ev.n + 31) // 32 * 32
    d = _device(ev, ld)
    f = _fitter(ev)
    out = f.outputs(ev.n, ld=ld)
    for k in ("par", "cov", "chi2"):
        out[k].fill_(float("nan"))
    bufs = dict(par_out=out["par"], cov_out=out["cov"], q_out=out["q"], chi2=out["chi2"],
                status=out["status"])
    if entry == "fit":
        f.run(*d, ev.ntrk, ev.mode, out=out)
    elif entry == "plan":
        plan = fit.fit_plan_create(f.h, ev.ntrk, ev.mode, NLAYER, persistent=False)
        fit.fit_plan_run(plan, *d, **bufs)
        torch.cuda.synchronize()
        fit.fit_plan_destroy(plan)
    elif entry == "noalloc":
        geo = [fit.Geometry(ev.B, s) for s in ev.surf]
        per_event = fit.fit_propagate_update_noalloc(geo[0], geo[1], *d, ev.ntrk, ev.mode, **bufs)
        for c, n, m in zip(per_event, ev.ntrk, ev.mode):  # one step a layer, seldom two
            assert n * NLAYER * (m == 0) <= c["iterations"] <= 2 * n * NLAYER * (m == 0)
        assert [c["tracks"] for c in per_event] == [int(n) for n in ev.ntrk]
    else:
        tiles = [a if k == 2 else torch.from_numpy(inputs.to_aosoa32(a.cpu().numpy(), ld)).cuda()
                 for k, a in enumerate(d)]
        fit.fit_propagate_update_layout(f.h, *tiles, ev.ntrk, ev.mode, fit.FIT_LAYOUT_AOSOA32, ld,
                                        out["par"], out["cov"], out["q"], out["chi2"],
                                        status=out["status"])
    if entry != "noalloc":
        assert f.sync()["tracks"] == ev.n
    got = {k: out[k].cpu().numpy() for k in ("par", "cov", "chi2", "q", "status")}
    if entry == "aosoa":
        for k in ("par", "cov"):
            got[k] = inputs.from_aosoa32(got[k].reshape(-1), got[k].shape, ev.n)
    f.close()
    _check(ev, {k: v[..., :ev.n] for k, v in got.items()}, entry)


# 303 runs: two tables of 128 a mode.  The kernels with one track per thread
# treat every track alone, so their results in event order are bit for bit
# those of the same tracks sorted by mode (two runs).
@pytest.mark.parametrize("entry", ["f64", "find", "find64", "adjoint", "seeded"])
def test_track_kernels_many_runs(entry):
    ev = _events(303)
    n, ld = ev.n, (ev.n + 3) // 4 * 4
    order = np.concatenate([_of_mode(ev, 0), _of_mode(ev, 1)])
    counts = [len(_of_mode(ev, 0)), len(_of_mode(ev, 1))]
    f = _fitter(ev)
    if entry == "seeded":
        m = fit.fit_mlp_create(0, seed=3)
        fit.fit_mlp_attach(f.h, m)
        torch.cuda.synchronize()
        fit.fit_mlp_destroy(m)
    dtype = torch.float64 if entry in ("f64", "find64") else torch.float32

    def run(nt, md, idx):
        par, cov, q, hpos, hcov = _device(ev, ld, dtype)
        if idx is not None:
            par, cov, q, hpos, hcov = (gpu_util.to_dev(a.cpu().numpy()[..., idx], ld)
                                       for a in (par, cov, q, hpos, hcov))
        out = f.outputs(n, ld=ld)
        o = {k: v.to(dtype) if v is not None and v.is_floating_point() else v for k, v in out.items()}
        args = (o["par"], o["cov"], o["q"], o["chi2"])
        res = [o["par"], o["cov"], o["q"], o["chi2"], o["status"]]
        if entry == "f64":
            fit.fit_propagate_update_f64(f.h, par, cov, q, hpos, hcov, nt, md, *args,
                                         status=o["status"])
        elif entry == "seeded":
            f.run(par, cov, q, hpos, hcov, nt, md, out=o)
        elif entry == "adjoint":
            tape = torch.empty(fit.fit_tape_bytes(NLAYER, ld) // 4, device="cuda")
            g = [torch.empty((NLAYER, 3, ld), device="cuda"), torch.empty((6, ld), device="cuda"),
                 torch.empty((21, ld), device="cuda")]
            fit.fit_adjoint_forward(f.h, par, cov, q, hpos, hcov, nt, md, tape, *args,
                                    status=o["status"])
            fit.fit_adjoint_backward(f.h, hpos, hcov, nt, md, tape, torch.ones(ld, device="cuda"), *g)
            res += g
        else:
            chosen = torch.empty((NLAYER, ld), dtype=torch.int8, device="cuda")
            fit.fit_find_tracks(f.h, par, cov, q, hpos[:, None].contiguous(),
                                hcov[:, None].contiguous(), nt, md, 30.0, chosen, *args,
                                status=o["status"])
            res.append(chosen)
        torch.cuda.synchronize()
        assert f.sync()["tracks"] == n
        return [r.cpu().numpy()[..., :n] for r in res]

    got = run(ev.ntrk, ev.mode, None)
    ref = run(counts, [0, 1], order)
    f.close()
    # the seeded handle's p2z tracks run in pairs, which the order changes
    keep = slice(0, counts[0]) if entry == "seeded" else slice(0, n)
    for a, b in zip(got, ref):
        np.testing.assert_array_equal(a[..., order][..., keep], b[..., keep])


# A call at or below a block of 128 tracks per SM runs one track per thread,
# a larger one pairs: the same operations with the same rounding.  Momenta
# whose turn per layer stays in the short series' range (|u| <= 0.1), so that
# no pair's range test depends on the partner.
@pytest.mark.parametrize("n", [1, 2, 127, 4097])
@pytest.mark.parametrize("entry", ["fit", "aosoa", "noalloc"])
def test_small_call_rounds_like_pairs(entry, n):
    big = torch.cuda.get_device_properties(0).multi_processor_count * 128 + 1
    sets = [inputs.generate(m, big, seed=67 + m, pt_range=(1.5, 10.0)) for m in (0, 1)]
    geo = [fit.Geometry(s.B, s.surf) for s in sets]
    f = fit.Fitter(*geo)

    def run(ts, k):
        ld = (k + 31) // 32 * 32
        d = [gpu_util.to_dev(np.ascontiguousarray(a[..., :k]), ld)
             for a in (ts.par0, ts.cov0, ts.q, ts.hpos, ts.hcov)]
        out = f.outputs(k, ld=ld, layers=True)
        bufs = dict(par_out=out["par"], cov_out=out["cov"], q_out=out["q"], chi2=out["chi2"],
                    chi2_layer=out["chi2_layer"], status=out["status"])
        if entry == "fit":
            f.run(*d, [k], [ts.mode], out=out)
        elif entry == "noalloc":
            fit.fit_propagate_update_noalloc(*geo, *d, [k], [ts.mode], **bufs)
        else:
            tiles = [a if i == 2 else torch.from_numpy(inputs.to_aosoa32(a.cpu().numpy(), ld)).cuda()
                     for i, a in enumerate(d)]
            fit.fit_propagate_update_layout(f.h, *tiles, [k], [ts.mode], fit.FIT_LAYOUT_AOSOA32, ld,
                                            out["par"], out["cov"], out["q"], out["chi2"],
                                            chi2_layer=out["chi2_layer"], status=out["status"])
        res = {i: v.cpu().numpy() for i, v in out.items()}
        if entry == "aosoa":
            for i in ("par", "cov", "chi2_layer"):
                res[i] = inputs.from_aosoa32(res[i].reshape(-1), res[i].shape, k)
        f.sync()
        return {i: v[..., :n] for i, v in res.items()}

    for ts in sets:
        small, pairs = run(ts, n), run(ts, big)
        whole = n & ~1  # the last of an odd count has no partner: the one-lane path
        for i in small:
            np.testing.assert_array_equal(small[i][..., :whole], pairs[i][..., :whole], err_msg=i)
    f.close()


@pytest.mark.parametrize("layout", [fit.FIT_LAYOUT_SOA, fit.FIT_LAYOUT_AOSOA32])
def test_default_plan_equals_the_persistent_form(layout):
    """A plan left at its default shape runs one launch per mode over the same
    pairs as the persistent form: bit for bit its results.  Odd event edges;
    more tracks than a small call has."""
    ev = inputs.generate_events(inputs.uneven_event_sizes(60, 83, median=600.0, hi=3000),
                                inputs.uneven_event_modes(60, 83), seed=83)
    assert ev.n > torch.cuda.get_device_properties(0).multi_processor_count * 128
    ld = (ev.n + 31) // 32 * 32
    d = _device(ev, ld)
    if layout == fit.FIT_LAYOUT_AOSOA32:
        d = [a if k == 2 else torch.from_numpy(inputs.to_aosoa32(a.cpu().numpy(), ld)).cuda().view(a.shape)
             for k, a in enumerate(d)]
    f = _fitter(ev)
    got = []
    for blocks_per_sm in (0, 3):
        out = f.outputs(ev.n, ld=ld, layers=True)
        plan = fit.fit_plan_create(f.h, ev.ntrk, ev.mode, NLAYER, blocks_per_sm=blocks_per_sm,
                                   layout=layout)
        for _ in range(2):  # captured, then replayed
            for k in ("par", "cov", "chi2", "chi2_layer"):
                out[k].fill_(float("nan"))
            fit.fit_plan_run(plan, *d, par_out=out["par"], cov_out=out["cov"], q_out=out["q"],
                             chi2=out["chi2"], chi2_layer=out["chi2_layer"], status=out["status"])
            torch.cuda.synchronize()
        fit.fit_plan_destroy(plan)
        got.append({k: v.cpu().numpy() for k, v in out.items()} | {"counters": f.sync()})
    f.close()
    assert got[0].pop("counters") == got[1].pop("counters")
    for k in got[0]:
        a, b = got[0][k], got[1][k]
        if a.ndim == 1:
            a, b = a[:ev.n], b[:ev.n]
        elif layout == fit.FIT_LAYOUT_SOA:
            a, b = a[:, :ev.n], b[:, :ev.n]
        np.testing.assert_array_equal(a, b, err_msg=k)


@pytest.mark.parametrize("ncand", [1, 2, 3, 4, 5, 7, 8, 13, 16])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_finder_choice_does_not_depend_on_the_number_of_slots(ncand, dtype):
    """Candidates pass through a few register slots, in one order or another by
    their number.  Each layer's own hit in a random one of ncand places, the
    others 1e3 cm away along z (p2r) or x (p2z), far beyond the gate: the
    finder takes the own hit and fits what one candidate alone gives, bit for
    bit."""
    n, ld = 301, 304
    g = torch.Generator().manual_seed(ncand)
    for mode in (0, 1):
        ts = inputs.generate(mode, n, seed=79)
        par, cov, q, hpos, hcov = (gpu_util.to_dev(a, ld) if k == 2 else gpu_util.to_dev(a, ld).to(dtype)
                                   for k, a in enumerate((ts.par0, ts.cov0, ts.q, ts.hpos, ts.hcov)))
        slot = torch.randint(0, ncand, (NLAYER, ld), generator=g).cuda()
        cpos, ccov = hpos[:, None].repeat(1, ncand, 1, 1), hcov[:, None].repeat(1, ncand, 1, 1)
        far = torch.arange(ncand, device="cuda")[None, :, None] != slot[:, None]
        cpos[:, :, 2 if mode == 0 else 0] += 1e3 * far
        f = fit.Fitter(*[fit.Geometry(ts.B, ts.surf) if m == mode else None for m in (0, 1)])

        def find(cp, cc):
            o = f.outputs(n, ld=ld)
            out = [o["par"].to(dtype), o["cov"].to(dtype), o["q"], o["chi2"].to(dtype)]
            chosen = torch.empty((NLAYER, ld), dtype=torch.int8, device="cuda")
            fit.fit_find_tracks(f.h, par, cov, q, cp, cc, [n], [mode], 1e4, chosen, *out)
            f.sync()
            return [r[..., :n] for r in out + [chosen]]

        one = find(hpos[:, None].contiguous(), hcov[:, None].contiguous())
        many = find(cpos, ccov)
        f.close()
        assert (one[4] == 0).all() and torch.equal(many[4].long(), slot[:, :n])
        for a, b in zip(one[:4], many[:4]):
            assert torch.equal(a, b)


@pytest.mark.parametrize("entry", ["fit", "find", "f64", "adjoint"])
@pytest.mark.parametrize("ntrk", [101, 13001])  # one launch or one for each mode, side by side
def test_calls_replay_from_a_captured_graph(entry, ntrk):
    """A call captured into a graph on the caller's stream holds its run tables
    and both modes' launches: replayed on new inputs in the same buffers it
    gives what the call gives."""
    nt, md = np.array([ntrk, ntrk, 3]), np.array([0, 1, 0], np.int32)
    evs = [inputs.generate_events(nt, md, seed=s, nlayer=NLAYER) for s in (101, 103)]
    n, ld = evs[0].n, (evs[0].n + 31) // 32 * 32
    dtype = torch.float64 if entry == "f64" else torch.float32
    d = _device(evs[0], ld, dtype)
    f = _fitter(evs[0])
    out = f.outputs(n, ld=ld)
    o = [out[k].to(dtype) if k != "q" else out[k] for k in ("par", "cov", "q", "chi2")]
    chosen = torch.empty((NLAYER, ld), dtype=torch.int8, device="cuda")
    tape = torch.empty(fit.fit_tape_bytes(NLAYER, ld) // 4, device="cuda")
    grads = [torch.empty((NLAYER, 3, ld), device="cuda"), torch.empty((6, ld), device="cuda"),
             torch.empty((21, ld), device="cuda")]
    w = torch.ones(ld, device="cuda")
    cand = [d[3][:, None].contiguous(), d[4][:, None].contiguous()]

    def call():
        if entry == "fit":
            fit.fit_propagate_update(f.h, *d, nt, md, *o)
        elif entry == "f64":
            fit.fit_propagate_update_f64(f.h, *d, nt, md, *o)
        elif entry == "find":
            fit.fit_find_tracks(f.h, *d[:3], *cand, nt, md, 30.0, chosen, *o)
        else:
            fit.fit_adjoint_forward(f.h, *d, nt, md, tape, *o)
            fit.fit_adjoint_backward(f.h, d[3], d[4], nt, md, tape, w, *grads)

    call()
    f.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    new = _device(evs[1], ld, dtype)
    for a, b in zip(d, new):
        a.copy_(b)
    cand[0].copy_(d[3][:, None])
    cand[1].copy_(d[4][:, None])
    results = []
    for run in (g.replay, call):
        for t in o + grads:
            t.fill_(7)
        torch.cuda.synchronize()
        run()
        torch.cuda.synchronize()
        results.append([t[..., :n].clone() for t in o + (grads if entry == "adjoint" else [])])
    f.sync()
    f.close()
    for a, b in zip(*results):
        assert torch.equal(a, b)
