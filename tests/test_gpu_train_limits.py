"""fit_mlp_train where its blocks do not all meet, and where they do not all fit
on the device: a training that gives up leaves the network as it was, and one
with two launches a step gives what one launch for all gives."""
import numpy as np
import pytest

from paper_2409_09228_gb300 import fit

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("needs a CUDA device", allow_module_level=True)

N, BATCH = 65536, 64  # 1024 steps: two launches


def _samples():
    g = torch.Generator().manual_seed(163)
    x = torch.randn((N, 8), generator=g)
    y = torch.tanh(x[:, 0] - 0.5 * x[:, 3]) * x[:, 5]
    return x.cuda(), y.cuda()


def _net(x, y):
    """A network that has been trained a little: nonzero moments and step."""
    m = fit.fit_mlp_create(0, seed=167)
    fit.fit_mlp_train(m, x[:4096], y[:4096], epochs=2, batch=512)
    return m


def _outputs(m, x):
    y = torch.empty(1000, device="cuda")
    fit.fit_mlp_forward(m, x[:1000], y)
    return y.cpu().numpy()


def test_a_training_that_gives_up_changes_nothing():
    x, y = _samples()
    a, b = _net(x, y), _net(x, y)
    params, out = fit.fit_mlp_get_params(a), _outputs(a, x)
    fit.fit_probe_train_limits(a, looks=0)  # a block whose first look is too early gives up
    with pytest.raises(fit.FitError) as e:
        fit.fit_mlp_train(a, x, y, epochs=1, batch=BATCH, beta1=0.7, beta2=0.9, eps=1e-4)
    assert e.value.code == fit.FIT_ERR_TIMEOUT
    np.testing.assert_array_equal(fit.fit_mlp_get_params(a), params)
    np.testing.assert_array_equal(_outputs(a, x), out)
    # its Adam state too: a step and a training go on as in a twin that never failed
    fit.fit_probe_train_limits(a)
    grad = torch.linspace(-1, 1, fit.FIT_MLP_PARAMS, device="cuda")
    res = []
    for m in (a, b):
        fit.fit_mlp_adam_step(m, grad, 1e-3)
        step = fit.fit_mlp_get_params(m)
        loss = fit.fit_mlp_train(m, x, y, epochs=1, batch=BATCH)
        res.append((step, loss, fit.fit_mlp_get_params(m), _outputs(m, x)))
        fit.fit_mlp_destroy(m)
    for p, q in zip(*res):
        np.testing.assert_array_equal(p, q)
    assert not np.array_equal(res[0][2], params)


def test_two_launches_a_step_give_the_same():
    """At most 38 blocks are taken to run together, one too few for a parameter
    a thread and the loss."""
    x, y = _samples()
    res = []
    for blocks in (0, 38):
        m = _net(x, y)
        fit.fit_probe_train_limits(m, blocks=blocks)
        loss = fit.fit_mlp_train(m, x[:40000], y[:40000], epochs=2, batch=1024)
        res.append((loss, fit.fit_mlp_get_params(m), _outputs(m, x)))
        fit.fit_mlp_destroy(m)
    for p, q in zip(*res):
        np.testing.assert_array_equal(p, q)
