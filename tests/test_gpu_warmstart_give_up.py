"""A convolution whose bounded wait runs out is reported by the network's calls, once,
and its results do not reach the weights.  The flags are set by a kernel of the
tests' own on the network's stream, as a kernel that gives up sets them; no wait is
made to run out."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1703_04446_gb300 import lgnk, synth

pytestmark = pytest.mark.gpu


@pytest.fixture()
def net():
    n = lgnk.WarmStart(16, 4, 2, 0.05)
    n.set_params(torch.from_numpy(synth.warmstart_init(4, 0)))
    yield n
    n.close()


def _give_up(net):
    net.lib.lgnk_internal_ws_give_up.argtypes = [ctypes.c_void_p]
    net.lib.lgnk_internal_ws_give_up(net.handle)


def _pairs():
    rng = np.random.default_rng(0)
    x = [torch.from_numpy(rng.uniform(size=(2, 16, 16)).astype(np.float32)).cuda() for _ in range(2)]
    return x + [torch.from_numpy(rng.normal(size=(2, 2, 8, 8)).astype(np.float32)).cuda()]


@pytest.mark.parametrize("call", ["predict", "train", "params", "grads"])
def test_the_next_call_reports_once(net, call):
    T, R, vt = _pairs()
    calls = {"predict": lambda: net.predict(T, R), "train": lambda: net.train_step(T, R, vt, 0.0, return_loss=False),
             "params": net.params, "grads": net.grads}
    v = net.predict(T, R).clone()
    _give_up(net)
    torch.cuda.synchronize()
    with pytest.raises(lgnk.LgnkError, match="gave up"):
        calls[call]()
    calls[call]()
    assert torch.equal(net.predict(T, R), v)


@pytest.mark.parametrize("with_loss", [False, True])
def test_weights_are_not_updated_from_an_unfinished_step(net, with_loss):
    T, R, vt = _pairs()
    p, v = net.params().clone(), net.predict(T, R).clone()
    torch.cuda.synchronize()
    torch.cuda._sleep(20_000_000)         # the flags are set after the step's call has begun
    _give_up(net)
    if with_loss:
        with pytest.raises(lgnk.LgnkError, match="gave up"):
            net.train_step(T, R, vt, 1e-2)
    else:
        net.train_step(T, R, vt, 1e-2, return_loss=False)
        torch.cuda.synchronize()
        with pytest.raises(lgnk.LgnkError, match="gave up"):
            net.params()
    assert torch.equal(net.params(), p)
    assert torch.equal(net.predict(T, R), v)
    net.train_step(T, R, vt, 1e-2)        # and the network works on
    assert not torch.equal(net.params(), p)


def test_new_parameters_are_used_whatever_happened_before(net):
    T, R, _ = _pairs()
    _give_up(net)
    torch.cuda.synchronize()
    net.set_params(torch.from_numpy(synth.warmstart_init(4, 1)))
    with pytest.raises(lgnk.LgnkError, match="gave up"):
        net.predict(T, R)
    other = lgnk.WarmStart(16, 4, 2, 0.05)
    other.set_params(torch.from_numpy(synth.warmstart_init(4, 1)))
    assert torch.equal(net.predict(T, R), other.predict(T, R))
    other.close()
