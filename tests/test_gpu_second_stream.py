"""The second stream that carries the p2z launches of a call with both modes:
calls on different streams and threads stay independent, and a capture on one
stream leaves calls on the others alone."""
import ctypes
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

from paper_2409_09228_gb300 import fit, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("needs a CUDA device", allow_module_level=True)

import gpu_util  # noqa: E402

NLAYER = 20
ENTRIES = ["fit", "aosoa", "plan", "mapped", "host", "f64", "find", "adjoint"]


class Calls:
    """One entry on events of both modes; a call writes outputs of its own."""

    def __init__(self, entry, seed=137):
        # more tracks than a small call has, fewer than an FP64 call that takes one stream
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        n = 28 * sms if entry == "f64" else 70 * sms
        self.entry, self.nt, self.md = entry, np.array([n, n]), np.array([0, 1], np.int32)
        ev = inputs.generate_events(self.nt, self.md, seed=seed, nlayer=NLAYER)
        self.n, self.ld = ev.n, (ev.n + 31) // 32 * 32
        self.f = fit.Fitter(fit.Geometry(ev.B, ev.surf[0]), fit.Geometry(ev.B, ev.surf[1]))
        d = [gpu_util.to_dev(a, self.ld) for a in (ev.par0, ev.cov0, ev.q, ev.hpos, ev.hcov)]
        if entry == "aosoa":
            d = [a if k == 2 else torch.from_numpy(inputs.to_aosoa32(a.cpu().numpy(), self.ld)).cuda()
                 for k, a in enumerate(d)]
        elif entry == "f64":
            d = [a if k == 2 else a.double() for k, a in enumerate(d)]
        elif entry in ("mapped", "host"):
            d = [a.cpu().pin_memory() for a in d]
        elif entry == "find":
            d[3:] = [a[:, None].contiguous() for a in d[3:]]
        self.d = d
        if entry == "plan":
            self.plan = fit.fit_plan_create(self.f.h, self.nt, self.md, NLAYER)

    def outputs(self):
        o = self.f.outputs(self.n, ld=self.ld)
        o = [o[k] for k in ("par", "cov", "q", "chi2")]
        if self.entry == "f64":
            o = [a if k == 2 else a.double() for k, a in enumerate(o)]
        elif self.entry in ("mapped", "host"):
            o = [a.cpu().pin_memory() for a in o]
        for a in o:
            a.fill_(7)
        o = {"out": o}
        if self.entry == "find":
            o["chosen"] = torch.zeros((NLAYER, self.ld), dtype=torch.int8, device="cuda")
        if self.entry == "adjoint":
            o["tape"] = torch.zeros(fit.fit_tape_bytes(NLAYER, self.ld) // 4, device="cuda")
            o["grads"] = [torch.zeros(s + (self.ld,), device="cuda") for s in ((NLAYER, 3), (6,), (21,))]
            o["weight"] = torch.ones(self.ld, device="cuda")
        return o

    def __call__(self, o, stream):
        f, d, nt, md, out = self.f, self.d, self.nt, self.md, o["out"]
        bufs = dict(zip(("par_out", "cov_out", "q_out", "chi2"), out), stream=stream)
        if self.entry == "fit":
            fit.fit_propagate_update(f.h, *d, nt, md, **bufs)
        elif self.entry == "aosoa":
            fit.fit_propagate_update_layout(f.h, *d, nt, md, fit.FIT_LAYOUT_AOSOA32, self.ld, **bufs)
        elif self.entry == "plan":
            fit.fit_plan_run(self.plan, *d, **bufs)
        elif self.entry == "mapped":
            fit.fit_propagate_update_mapped(f.h, *d, nt, md, **bufs)
        elif self.entry == "host":
            fit.fit_propagate_update_host(f.h, *d, nt, md, **bufs)
        elif self.entry == "f64":
            fit.fit_propagate_update_f64(f.h, *d, nt, md, **bufs)
        elif self.entry == "find":
            fit.fit_find_tracks(f.h, *d, nt, md, 30.0, o["chosen"], **bufs)
        else:
            fit.fit_adjoint_forward(f.h, *d, nt, md, o["tape"], **bufs)
            fit.fit_adjoint_backward(f.h, d[3], d[4], nt, md, o["tape"], o["weight"], *o["grads"],
                                     stream=stream)

    def results(self, o):
        r = o["out"] + o.get("grads", [])
        return r if self.entry == "aosoa" else [a[..., :self.n] for a in r]

    def reference(self):
        o = self.outputs()
        torch.cuda.synchronize()
        self(o, torch.cuda.current_stream())
        torch.cuda.synchronize()
        return self.results(o)

    def same(self, o, ref):
        return all(torch.equal(a, b) for a, b in zip(self.results(o), ref))

    def close(self):
        torch.cuda.synchronize()
        if self.entry == "plan":
            fit.fit_plan_destroy(self.plan)
        self.f.close()


@pytest.mark.parametrize("entry", ENTRIES)
def test_a_capture_leaves_other_streams_alone(entry):
    """While a call of both modes is being captured on one stream, the same
    call on another runs; the captured one replays."""
    c = Calls(entry)
    ref = c.reference()
    o = [c.outputs() for _ in range(2)]
    other = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        c(o[0], torch.cuda.current_stream())
        c(o[1], other)
    torch.cuda.synchronize()
    assert c.same(o[1], ref) and not c.same(o[0], ref)
    g.replay()
    torch.cuda.synchronize()
    assert c.same(o[0], ref)
    c.close()


@pytest.mark.parametrize("entry", ["fit", "find"])
def test_more_streams_than_second_streams(entry):
    """Calls on twenty streams, all of them held up at first, so that each
    finds the earlier ones' second streams at work."""
    c = Calls(entry)
    ref = c.reference()
    streams = [torch.cuda.Stream() for _ in range(20)]
    o = [c.outputs() for _ in streams]
    torch.cuda.synchronize()
    for s in streams:
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)  # ~10 ms
    for s, x in zip(streams, o):
        c(x, s)
    torch.cuda.synchronize()
    assert all(c.same(x, ref) for x in o)
    c.close()


@pytest.mark.parametrize("entry", ["fit", "adjoint"])
def test_calls_from_several_threads(entry):
    """Four host threads on one handle, two of them on the same stream."""
    c = Calls(entry)
    ref = c.reference()
    s = [torch.cuda.Stream() for _ in range(3)]
    jobs = [(st, [c.outputs() for _ in range(8)]) for st in (s[0], s[0], s[1], s[2])]
    torch.cuda.synchronize()
    errors = []

    def work(stream, outs):
        try:
            for o in outs:
                c(o, stream)
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(e)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    assert all(c.same(o, ref) for _, outs in jobs for o in outs)
    c.close()


@pytest.mark.parametrize("entry", ["fit", "plan", "aosoa"])
def test_the_modes_run_side_by_side(entry):
    """40000 tracks of each mode, one block of either an SM: the two launches
    share the SMs, so that a call takes well under the sum of its modes' times
    (graphs of the calls alone, so that no host time counts; 0.72 measured,
    1.0 where one launch waits for the other)."""
    n = 40000
    ev = inputs.generate_events([n, n], [0, 1], seed=179, nlayer=NLAYER)
    f = fit.Fitter(fit.Geometry(ev.B, ev.surf[0]), fit.Geometry(ev.B, ev.surf[1]))
    best = {}
    for name, nt, md, part in (("r", [n], [0], slice(0, n)), ("z", [n], [1], slice(n, 2 * n)),
                               ("both", [n, n], [0, 1], slice(0, 2 * n))):
        total = sum(nt)
        d = [gpu_util.to_dev(np.ascontiguousarray(a[..., part]), total)
             for a in (ev.par0, ev.cov0, ev.q, ev.hpos, ev.hcov)]
        if entry == "aosoa":
            d = [a if k == 2 else torch.from_numpy(inputs.to_aosoa32(a.cpu().numpy(), total)).cuda()
                 for k, a in enumerate(d)]
        o = f.outputs(total, ld=total)
        bufs = dict(par_out=o["par"], cov_out=o["cov"], q_out=o["q"], chi2=o["chi2"])
        plan = fit.fit_plan_create(f.h, nt, md, NLAYER)

        def call():
            if entry == "plan":
                fit.fit_plan_run(plan, *d, **bufs)
            elif entry == "fit":
                fit.fit_propagate_update(f.h, *d, nt, md, **bufs)
            else:
                fit.fit_propagate_update_layout(f.h, *d, nt, md, fit.FIT_LAYOUT_AOSOA32, total, **bufs)

        call()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(20):
                call()
        times = []
        for _ in range(8):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            g.replay()
            e[1].record()
            torch.cuda.synchronize()
            times.append(e[0].elapsed_time(e[1]) / 20)
        best[name] = min(times)
        fit.fit_plan_destroy(plan)
    f.close()
    assert best["both"] < 0.87 * (best["r"] + best["z"]), best


def independent(entry):
    """In a process of its own (few streams, a hardware queue for each): a call
    on stream b ends while stream a, which has a call queued, is held up."""
    rt = ctypes.CDLL("libcudart.so.13")
    torch.zeros(1, device="cuda")

    def new_stream():
        h = ctypes.c_void_p()
        assert rt.cudaStreamCreateWithFlags(ctypes.byref(h), 1) == 0
        return torch.cuda.ExternalStream(h.value)

    c = Calls(entry)
    ref = c.reference()
    a, b = new_stream(), new_stream()
    o = [c.outputs() for _ in range(4)]
    c(o[2], a)
    c(o[3], b)
    torch.cuda.synchronize()
    held, done = torch.cuda.Event(), torch.cuda.Event()
    with torch.cuda.stream(a):
        torch.cuda._sleep(1_000_000_000)  # ~0.5 s
        held.record(a)
    c(o[0], a)
    c(o[1], b)
    done.record(b)
    done.synchronize()
    still_held = not held.query()
    torch.cuda.synchronize()
    assert all(c.same(x, ref) for x in o)
    c.close()
    assert still_held, "the call on stream b waited for stream a"


@pytest.mark.parametrize("entry", ["fit", "plan", "find", "adjoint", "f64", "mapped"])
def test_a_stalled_stream_holds_up_no_other(entry):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, os.path.abspath(__file__), entry], capture_output=True,
                       text=True, timeout=300, cwd=root,
                       env={**os.environ, "CUDA_DEVICE_MAX_CONNECTIONS": "32", "PYTHONPATH": root})
    assert r.returncode == 0, r.stdout + r.stderr


if __name__ == "__main__":
    independent(sys.argv[1])
