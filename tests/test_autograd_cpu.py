"""The autograd function of fit.chi2 with the library's calls replaced by
stand-ins (no GPU): what reaches the reverse sweep, and what comes back."""
import pytest

from paper_2409_09228_gb300 import fit

torch = pytest.importorskip("torch")

NLAYER, LD = 3, 8


class Fitter:
    h = 0

    def outputs(self, n, ld):
        return {"par": torch.zeros(6, ld), "cov": torch.zeros(21, ld),
                "q": torch.zeros(ld, dtype=torch.int32), "chi2": torch.zeros(ld),
                "status": torch.zeros(ld, dtype=torch.uint8)}


class NoGradient(torch.autograd.Function):
    """Returns an undefined gradient for its first input."""

    @staticmethod
    def forward(ctx, a, b):
        return a.sum() + b.sum()

    @staticmethod
    def backward(ctx, g):
        return None, g.expand(LD)


@pytest.fixture
def calls(monkeypatch):
    """A reverse sweep that returns its chi2 gradient for every gradient."""
    def backward(h, hpos, hcov, ntrk, mode, tape, grad_chi2, *out, stream=None):
        assert grad_chi2.is_contiguous() and grad_chi2.dtype == torch.float32
        for g in out:
            g.copy_(grad_chi2.expand(g.shape))

    monkeypatch.setattr(fit, "fit_tape_bytes", lambda nlayer, ld: 4)
    monkeypatch.setattr(fit, "fit_adjoint_forward", lambda *a, **k: None)
    monkeypatch.setattr(fit, "fit_adjoint_backward", backward)


def _chi2():
    leaves = [torch.zeros(s + (LD,), requires_grad=True) for s in ((NLAYER, 3), (6,), (21,))]
    hcov = torch.zeros(NLAYER, 6, LD)
    return leaves, fit.chi2(Fitter(), *leaves, torch.ones(LD, dtype=torch.int32), hcov, [5], [0])


def test_gradient_of_a_weighted_sum(calls):
    leaves, (chi2, _, _) = _chi2()
    w = torch.arange(LD, dtype=torch.float32)
    for g in torch.autograd.grad((w * chi2).sum(), leaves):
        assert torch.equal(g, w.expand(g.shape))


def test_undefined_gradient_is_zero(calls):
    """Where what follows chi2 returns no gradient for it, the inputs' are
    zeros, not missing."""
    leaves, (chi2, _, _) = _chi2()
    other = torch.zeros(LD, requires_grad=True)
    for g, x in zip(torch.autograd.grad(NoGradient.apply(chi2, other), leaves), leaves):
        assert g.shape == x.shape and (g == 0).all()
