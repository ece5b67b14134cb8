"""Which host buffers fit_propagate_update_host reads and writes in place: those
that a kernel may dereference throughout, without a race.  The decision alone;
no kernel runs on a buffer that it refuses."""
import ctypes

import numpy as np
import pytest

from paper_2409_09228_gb300 import fit

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("needs a CUDA device", allow_module_level=True)

PAGE, NLAYER, N = 1 << 16, 20, 4096  # a row of N floats: a quarter of PAGE

SHAPES = {"par_in": (6,), "cov_in": (21,), "q_in": (), "hpos": (NLAYER, 3), "hcov": (NLAYER, 6),
          "par_out": (6,), "cov_out": (21,), "q_out": (), "chi2": (), "chi2_layer": (NLAYER,),
          "status": ()}


def _pinned():
    return {k: torch.zeros(s + (N,), dtype=torch.uint8 if k == "status" else torch.int32 if k[0] == "q"
                           else torch.float32).pin_memory() for k, s in SHAPES.items()}


def _in_place(bufs):
    return fit.fit_probe_host_in_place(**bufs, n=N)


def _pageable(shape):
    """A float array that starts on a page of PAGE bytes, inside a larger one."""
    raw = np.zeros(4 * int(np.prod(shape)) + 3 * PAGE, np.uint8)
    skip = -raw.ctypes.data % PAGE + PAGE
    return raw[skip:skip + 4 * int(np.prod(shape))].view(np.float32).reshape(shape)


class _Locked:
    """Pieces (offset, bytes) of an array, each page-locked by itself."""

    def __init__(self, a, pieces):
        self.rt, self.at = ctypes.CDLL("libcudart.so.13"), [a.ctypes.data + o for o, _ in pieces]
        for p, (_, b) in zip(self.at, pieces):
            assert self.rt.cudaHostRegister(ctypes.c_void_p(p), ctypes.c_size_t(b), 2) == 0

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        for p in self.at:
            self.rt.cudaHostUnregister(ctypes.c_void_p(p))


def test_page_locked_throughout_is_taken_in_place():
    bufs = _pinned()
    assert _in_place(bufs)
    assert _in_place({**bufs, "chi2_layer": None, "status": None})
    a = _pageable((24, N))  # one registration, whole and larger than the array
    with _Locked(a, [(0, a.nbytes)]):
        assert _in_place({**bufs, "cov_in": a[:21]})
    assert not _in_place({**bufs, "cov_in": a[:21]})


@pytest.mark.parametrize("name", ["cov_in", "cov_out", "hcov", "chi2_layer"])
def test_arrays_locked_in_pieces_are_staged(name):
    """The head and the tail of an array are page-locked, or all of it in two
    registrations, or all but its last bytes: not one range, so not in place."""
    bufs = _pinned()
    a = _pageable(SHAPES[name] + (N,))
    assert a.nbytes > 4 * PAGE
    tail = (a.nbytes - 1) // PAGE * PAGE
    for pieces in ([(0, PAGE), (tail, a.nbytes - tail)], [(0, 2 * PAGE), (2 * PAGE, a.nbytes - 2 * PAGE)],
                   [(0, tail)]):
        with _Locked(a, pieces):
            assert not _in_place({**bufs, name: a})


def test_outputs_over_other_inputs_are_staged():
    """In place an output may only be the input it replaces: shifted, narrower
    or over another array, threads would overwrite what others have yet to
    read."""
    bufs = _pinned()
    own = {k: bufs[k.replace("out", "in")] for k in ("par_out", "cov_out", "q_out")}
    assert _in_place({**bufs, **own})
    wide = torch.zeros((30, N + 8)).pin_memory()  # ld of the inputs and the outputs: N + 8
    par = {"par_in": wide[:6], "cov_in": bufs["cov_in"].new_zeros((21, N + 8)).pin_memory(),
           "cov_out": torch.zeros((21, N + 8)).pin_memory()}
    assert _in_place({**bufs, **par, "par_out": wide[:6]})
    assert _in_place({**bufs, **par, "par_out": wide[6:12]})
    assert not _in_place({**bufs, **par, "par_out": wide[1:7]})
    assert not _in_place({**bufs, **par, "par_out": wide.view(-1)[4:].as_strided((6, N + 8), (N + 8, 1))})
    narrow = {**bufs, "par_out": bufs["par_in"].view(-1)[:6 * (N - 8)].view(6, N - 8)}
    assert not fit.fit_probe_host_in_place(**narrow, n=N - 8)
    assert not _in_place({**bufs, "chi2": bufs["hpos"][0, 0]})
    assert not _in_place({**bufs, "chi2_layer": bufs["hcov"].view(-1)[:NLAYER * N].view(NLAYER, N)})
