"""Plans whose events make more runs than a launch's tables hold, replayed on
new inputs; calls that fill a run table and take another launch."""
import ctypes

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
TABLE = 1024  # pair runs of a launch's table (lone tracks: twice as many)
SMALL_RUNS = 256  # pair runs of a mode that a small call's one launch holds (lone tracks: twice)


def runs(nt, md, m):
    """(pair runs, lone tracks) of mode m: its maximal runs of consecutive
    events as pairs that start at even tracks, and what their odd edges leave."""
    pairs = lone = 0
    start = np.concatenate([[0], np.cumsum(nt)])
    e = 0
    while e < len(nt):
        e0 = e
        while e < len(nt) and md[e] == md[e0]:
            e += 1
        t0, t1 = int(start[e0]), int(start[e])
        if md[e0] == m and t1 > t0:
            p0, p1 = (t0 + 1) & ~1, t1 & ~1
            pairs += p1 > p0
            lone += (t0 & 1) + ((t1 & 1) and t1 > p0)
    return pairs, lone


def _device(ev, ld):
    return [gpu_util.to_dev(a, ld) for a in (ev.par0, ev.cov0, ev.q, ev.hpos, ev.hcov)]


def _fitter(ev):
    return fit.Fitter(fit.Geometry(ev.B, ev.surf[0]), fit.Geometry(ev.B, ev.surf[1]))


def test_small_per_mode_plan_with_many_runs_replays_both_modes():
    """A plan of one launch per mode on few tracks in many runs: every run of
    the captured graph fits both modes' tracks on what the buffers then hold,
    bit for bit as one call does, and counts them."""
    nt = np.full(1400, 3)
    md = (np.arange(1400) % 2).astype(np.int32)
    assert min(runs(nt, md, m)[0] for m in (0, 1)) > SMALL_RUNS
    assert nt.sum() <= 128 * torch.cuda.get_device_properties(0).multi_processor_count
    evs = [inputs.generate_events(nt, md, seed=s, nlayer=NLAYER) for s in (107, 109, 113)]
    n = evs[0].n
    ld = gpu_util.pad_ld(n)
    f = _fitter(evs[0])
    d = _device(evs[0], ld)
    out = f.outputs(n, ld=ld, layers=True)
    plan = fit.fit_plan_create(f.h, nt, md, NLAYER, persistent=False)
    for ev in evs:  # captured by the first, replayed by the others
        for a, b in zip(d, _device(ev, ld)):
            a.copy_(b)
        for k, v in out.items():
            v.fill_(float("nan") if v.is_floating_point() else 77)
        torch.cuda.synchronize()
        fit.fit_plan_run(plan, *d, par_out=out["par"], cov_out=out["cov"], q_out=out["q"],
                         chi2=out["chi2"], chi2_layer=out["chi2_layer"], status=out["status"])
        got_counts = f.sync()
        ref = f.run(*d, nt, md, layers=True)
        ref_counts = f.sync()
        assert got_counts == ref_counts and got_counts["tracks"] == n
        for k in ref:
            assert torch.equal(out[k][..., :n], ref[k][..., :n]), k
    fit.fit_plan_destroy(plan)
    f.close()


def test_tuning_does_not_take_shapes_timed_on_older_kernels(tmp_path):
    """A cache entry of the key's third version was timed on a per-mode form
    that has changed since: it is measured anew, and the new entry is taken."""
    cache = str(tmp_path / "tune.txt")
    f = None
    info = {}
    for n in (1001, 1002):  # two keys that differ in the number of tracks alone
        ev = inputs.generate_events([n], [0], seed=127, nlayer=NLAYER)
        ld = gpu_util.pad_ld(n)
        f = f or _fitter(ev)
        out = f.outputs(n, ld=ld)
        plan = fit.fit_plan_create(f.h, [n], [0], NLAYER)
        info[n] = fit.fit_plan_tune(plan, *_device(ev, ld), out["par"], out["cov"], out["q"],
                                    out["chi2"], status=out["status"], cache_path=cache)
        fit.fit_plan_destroy(plan)
        line = open(cache).read()
        key, shape = line.split("\n")[-2].split("\t")
        assert f"tracks={n},0;" in key
        if n == 1001:
            old = key.replace("tracks=1001,0;", "tracks=1002,0;").split(";")
            old[1] = "v3"
            open(cache, "a").write(";".join(old) + "\t" + shape + "\n")
    f.close()
    assert info[1001]["tuned"] == info[1002]["tuned"] == 1


def test_failed_tuning_leaves_the_plan_as_it_was():
    """Tuning waits for its stream, which a stream under capture refuses: the
    call fails in its first candidate, and the plan keeps its shape and layout
    and runs as before."""
    ev = inputs.generate_events([300, 301], [0, 1], seed=131, nlayer=NLAYER)
    ld = (ev.n + 31) // 32 * 32
    f = _fitter(ev)
    d = _device(ev, ld)
    out = f.outputs(ev.n, ld=ld)
    bufs = dict(par_out=out["par"], cov_out=out["cov"], q_out=out["q"], chi2=out["chi2"],
                status=out["status"])
    plan = fit.fit_plan_create(f.h, ev.ntrk, ev.mode, NLAYER, threads_per_block=64, blocks_per_sm=2,
                               layout=fit.FIT_LAYOUT_TUNE)
    before = fit.fit_plan_get_info(plan)
    rt = ctypes.CDLL("libcudart.so.13")
    stream, graph = torch.cuda.Stream(), ctypes.c_void_p()
    torch.cuda.synchronize()
    assert rt.cudaStreamBeginCapture(ctypes.c_void_p(stream.cuda_stream), 2) == 0  # relaxed mode
    try:
        with pytest.raises(fit.FitError):
            fit.fit_plan_tune(plan, *d, stream=stream, **bufs)
    finally:  # whatever was captured is dropped unlaunched
        rt.cudaStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph))
        if graph.value:
            rt.cudaGraphDestroy(graph)
        rt.cudaGetLastError()
    assert fit.fit_plan_get_info(plan) == before
    ref = f.run(*d, ev.ntrk, ev.mode)
    fit.fit_plan_run(plan, *d, **bufs)
    torch.cuda.synchronize()
    fit.fit_plan_destroy(plan)
    f.close()
    np.testing.assert_allclose(out["par"][:, :ev.n].cpu().numpy(), ref["par"][:, :ev.n].cpu().numpy(),
                               rtol=1e-4, atol=1e-4)


def test_info_tells_the_default_form_from_a_persistent_shape():
    """A plan at its default shape runs one launch per mode and reports
    blocks_per_sm 0, the value that asks for it; a persistent shape reports
    the blocks per SM it launches."""
    f = fit.Fitter(fit.Geometry(3.8, inputs.surfaces(0)), None)
    blocks = {}
    for name, kw in (("default", {}), ("given", dict(blocks_per_sm=2)),
                     ("most", dict(threads_per_block=64))):
        plan = fit.fit_plan_create(f.h, [5000], [0], NLAYER, **kw)
        info = fit.fit_plan_get_info(plan)
        blocks[name] = info["blocks_per_sm"]
        assert info["persistent"] and info["items"] > 0 and info["tuned"] == 0
        fit.fit_plan_destroy(plan)
    f.close()
    assert blocks["default"] == 0 and blocks["given"] == 2 and blocks["most"] > 2


# Sizes that fill a launch's tables: three tracks an event give each run a pair
# and a lone track; events of two from an odd start give two lone tracks each.
FULL = {"pairs": np.full(2300, 3), "lone": np.concatenate([[1], np.full(2299, 2)])}


@pytest.mark.parametrize("fills", FULL)
@pytest.mark.parametrize("entry", ["fit", "noalloc", "plan", "per_mode"])
def test_a_full_run_table_takes_another_launch(entry, fills):
    nt, md = FULL[fills], (np.arange(len(FULL[fills])) % 2).astype(np.int32)
    for m in (0, 1):
        pairs, lone = runs(nt, md, m)
        assert pairs > TABLE if fills == "pairs" else lone > 2 * TABLE
    ev = inputs.generate_events(nt, md, seed=173, nlayer=NLAYER)
    ld = gpu_util.pad_ld(ev.n)
    f = _fitter(ev)
    d = _device(ev, ld)
    out = f.outputs(ev.n, ld=ld)
    for v in out.values():
        if v is not None:
            v.fill_(float("nan") if v.is_floating_point() else 77)
    bufs = dict(par_out=out["par"], cov_out=out["cov"], q_out=out["q"], chi2=out["chi2"],
                status=out["status"])
    if entry == "fit":
        f.run(*d, nt, md, out=out)
    elif entry == "noalloc":
        geo = [fit.Geometry(ev.B, s) for s in ev.surf]
        counts = fit.fit_propagate_update_noalloc(*geo, *d, nt, md, **bufs)
        for c, n, m in zip(counts, nt, md):
            assert c["tracks"] == n and n * NLAYER * (m == 0) <= c["iterations"] <= 2 * n * NLAYER * (m == 0)
    else:
        plan = fit.fit_plan_create(f.h, nt, md, NLAYER, persistent=entry == "plan")
        fit.fit_plan_run(plan, *d, **bufs)
        torch.cuda.synchronize()
        fit.fit_plan_destroy(plan)
    if entry != "noalloc":
        counts = f.sync()
        assert counts["tracks"] == ev.n
        assert nt[md == 0].sum() * NLAYER <= counts["iterations"] <= 2 * nt[md == 0].sum() * NLAYER
    got = {k: out[k][..., :ev.n].cpu().numpy() for k in ("par", "cov", "chi2", "q", "status")}
    f.close()
    mode = np.repeat(md, nt)
    for m in (0, 1):
        idx = np.nonzero(mode == m)[0]
        ts = inputs.TrackSet(m, ev.B, ev.surf[m], *(np.ascontiguousarray(a[..., idx]) for a in
                                                    (ev.par0, ev.cov0, ev.q, ev.hpos, ev.hcov)))
        parity.check({k: v[..., idx] for k, v in got.items()}, oracle.fit_set(ts), f"{entry} {fills} {m}")
