"""The inner products and step lengths of the device-side PCG loop, at the sizes
where the sums change form: one partial sum, 32 (one warp adds them) and 33 (the
block does), more than a block has threads, and vectors that several elements a
thread share, with the fused end of the product (diffusion) and without it.

The reference is the same three iterations with the product and the
preconditioner called through the API and every scalar in FP64 on the host.
Tolerance: the two differ by FP32 roundings of the vectors only, about ten a
component and iteration, amplified by at most the preconditioned system's
condition number (below 100 here): 3 * 10 * 6e-8 * 100 = 2e-4 of the solution."""
import numpy as np
import pytest
import torch

from tests._cases import rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vm", [(8, 8), (64, 64), (64, 66), (13, 11, 9), (48, 44, 40)])
@pytest.mark.parametrize("reg", ["diffusion", "curvature"])
def test_pcg_loop_matches_host_scalars(vm, reg):
    from paper_1703_04446_gb300 import lgnk
    d = len(vm)
    im = tuple(2 * a for a in vm)
    ctx = lgnk.Context(lgnk.Problem(image_m=im, velocity_m=vm, time_nodes=1, rk4_steps=2, regularizer=reg,
                                    alpha=1e-2, gamma=1e-2))
    x = np.meshgrid(*[(np.arange(m) + 0.5) / m for m in reversed(im)], indexing="ij")
    T = torch.from_numpy(np.exp(-8.0 * sum((c - 0.5) ** 2 for c in x)).astype(np.float32)).cuda()
    R = torch.from_numpy(np.exp(-9.0 * sum((c - 0.53) ** 2 for c in x)).astype(np.float32)).cuda()
    v0 = torch.zeros((1, d) + tuple(reversed(vm)), device="cuda")

    dot = lambda a, b: float((a.double() * b.double()).sum())
    g = ctx.objective(v0, T, R, grad=True)[3]
    r = -g
    z = ctx.precond(r)
    p, rz, xs = z.clone(), dot(r, z), torch.zeros_like(v0)
    for _ in range(3):
        Hp = ctx.hessvec(v0, T, p)
        a = rz / dot(p, Hp)
        xs, r = xs + a * p, r - a * Hp
        z = ctx.precond(r)
        b, rz = dot(r, z) / rz, dot(r, z)
        p = z + b * p

    v, rep = ctx.solve(T, R, None, max_gn=1, max_pcg=3, pcg_rtol=1e-12, gn_grad_rtol=0.0, matvec=0)
    ctx.close()
    assert rep["pcg_iters"] == 3
    v, xs = (t.cpu().numpy().astype(np.float64) for t in (v, xs))
    t = float((v * xs).sum() / (xs * xs).sum())
    step = 2.0 ** round(np.log2(t))           # the line search halves from 1
    assert step <= 1.0
    assert rel(v, step * xs) <= 2e-4
