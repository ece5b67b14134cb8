"""The FP64 kernels' small-angle series and quick reciprocals against their
general forms: fits whose angles, steps and magnitudes fall on either side of
each range, against the FP64 oracle."""
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


def _fit64(ts):
    ld = gpu_util.pad_ld(ts.n)
    d = [gpu_util.to_dev(a, ld) for a in (ts.par0, ts.cov0, ts.q, ts.hpos, ts.hcov)]
    d = [a if k == 2 else a.double() for k, a in enumerate(d)]
    geo = fit.Geometry(ts.B, ts.surf, tol=1e-12)
    f = fit.Fitter(geo if ts.mode == 0 else None, geo if ts.mode == 1 else None)
    o = f.outputs(ts.n, ld=ld)
    par, cov, chi2 = (o[k].double() for k in ("par", "cov", "chi2"))
    fit.fit_propagate_update_f64(f.h, *d, [ts.n], [ts.mode], par, cov, o["q"], chi2,
                                 status=o["status"])
    torch.cuda.synchronize()
    f.close()
    got = {"par": par, "cov": cov, "chi2": chi2, "q": o["q"], "status": o["status"]}
    return {k: v.cpu().numpy()[..., :ts.n] for k, v in got.items()}


# Layer spacings and momenta that turn a track by u = kappa h / 2 between
# surfaces from zero and far below the series' 1/4 (20 layers) over about it
# (8) to beyond it (4), with the updates' changes of angle around 1/16.
# Tolerances as test_gpu_f64.py's for 20 layers; wide layers shrink the 1/pT
# variance up to ~170-fold an update, which costs it that factor of relative
# precision.
@pytest.mark.parametrize("mode", [inputs.MODE_R, inputs.MODE_Z], ids=["p2r", "p2z"])
@pytest.mark.parametrize("nlayer,B,pt", [(20, 3.8, (0.7, 10.0)), (20, 0.0, (1.0, 2.0)),
                                         (8, 3.8, (0.7, 1.0)), (4, 3.8, (0.5, 0.8))])
def test_ranges_of_the_series(mode, nlayer, B, pt):
    ts = inputs.generate(mode, 700, seed=71, nlayer=nlayer, B=max(B, 1e-30), pt_range=pt)
    ts.B = float(np.float32(B))  # what the library and the oracle both take
    wide = 1.0 if nlayer == 20 else 170.0
    parity.check(_fit64(ts), oracle.fit_set(ts), f"mode {mode} {nlayer} layers B {B}",
                 rtol=1e-11 * wide, chi2_abs=1e-10 * wide)
