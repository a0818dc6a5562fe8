"""The layouts of a call in one launch: every call packs its own inputs and clears
its own sums, whatever ran before on the context.  Calls in mixed order on one
context, with inputs that change from call to call, against each call on a
context of its own, for sizes with one and with several blocks a part.

Tolerance: the same kernels on the same inputs; only the order of the atomic
additions differs, a few FP32 roundings of the sums (1e-6)."""
import numpy as np
import pytest
import torch

from tests._cases import rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("im,vm", [((12, 10), (6, 5)), ((70, 45), (33, 24)), ((26, 22, 18), (13, 11, 9))])
@pytest.mark.parametrize("model,K", [("transport", 1), ("transport", 3), ("continuity", 1), ("continuity", 3)])
def test_mixed_calls_match_fresh_contexts(im, vm, model, K):
    from paper_1703_04446_gb300 import lgnk
    d = len(im)
    prob = dict(image_m=im, velocity_m=vm, time_nodes=K, rk4_steps=5, model=model, regularizer="diffusion",
                alpha=1e-2, gamma=1e-3)
    rng = np.random.default_rng(5)
    img = lambda: torch.from_numpy(rng.uniform(size=tuple(reversed(im))).astype(np.float32)).cuda()
    vel = lambda: torch.from_numpy(0.03 * rng.normal(size=(K, d) + tuple(reversed(vm))).astype(np.float32)).cuda()
    calls = [("forward", lambda c, v, T, dv, r: [c.forward(v, T)]),
             ("hessvec", lambda c, v, T, dv, r: [c.hessvec(v, T, dv)]),
             ("jtvp", lambda c, v, T, dv, r: [c.jtvp(v, T, r)]),
             ("objective", lambda c, v, T, dv, r: [c.objective(v, T, r, grad=True)[3]]),
             ("jvp", lambda c, v, T, dv, r: [c.jvp(v, T, dv)]),
             ("value", lambda c, v, T, dv, r: [torch.tensor(c.objective(v, T, r))]),
             ("determinant", lambda c, v, T, dv, r: [c.jacobian_determinant(v, T)[0]])]
    shared = lgnk.Context(lgnk.Problem(**prob))
    for k in rng.permutation(2 * len(calls)):
        name, call = calls[k % len(calls)]
        args = (vel(), img(), vel(), img())
        own = lgnk.Context(lgnk.Problem(**prob))
        for got, want in zip(call(shared, *args), call(own, *args)):
            got, want = (t.cpu().numpy().astype(np.float64) for t in (got, want))
            assert rel(got, want) <= 1e-6, name
        own.close()
    shared.close()
