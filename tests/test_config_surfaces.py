"""What a Geometry takes as its surfaces (no GPU): a sequence of numbers, each
converted by float()."""
import numpy as np
import pytest

from paper_2409_09228_gb300 import fit

torch = pytest.importorskip("torch")


class Number:
    def __init__(self, v):
        self.v = v

    def __float__(self):
        return self.v


VALUES = [4.0, 9.578947, 15.1578951, 1e30, 1e-42]


@pytest.mark.parametrize("surf", [VALUES, tuple(VALUES), np.array(VALUES), np.array(VALUES, np.float32),
                                  np.repeat(VALUES, 2)[::2], np.array(VALUES, np.float64).astype(">f8"),
                                  [Number(v) for v in VALUES], [torch.tensor(v, dtype=torch.float64,
                                                                             requires_grad=True)
                                                                for v in VALUES],
                                  torch.tensor(VALUES, dtype=torch.float64), ["4", "9.578947"]],
                         ids=lambda s: type(s).__name__)
def test_accepted(surf):
    cfg, arr = fit._config(fit.Geometry(3.8, surf))
    assert cfg.nlayer == len(surf) == len(arr)
    assert list(arr) == [float(np.float32(float(v))) for v in surf]


@pytest.mark.parametrize("surf", [np.ones((2, 3)), [[4.0, 5.0], [6.0, 7.0]], [4.0, None], np.float32(4.0)],
                         ids=["2d", "nested", "none", "scalar"])
def test_refused(surf):
    with pytest.raises(TypeError):
        fit._config(fit.Geometry(3.8, surf))
