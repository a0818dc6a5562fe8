"""The mass-preserving adjoint adds w_c mu to each corner of a velocity cell: a corner
with a small weight keeps its relative accuracy (as a difference of the block's
moments it would be wrong by a rounding of mu, whatever its weight).

One voxel with mass near the upper corner of a coarse velocity cell, v = 0 and a
linear r: J^T r is (d_v I)^T of one vector, each node the product of its weight.
Tolerance: the node's value over the sum of all nodes against the exact weight, 2e-6
relative (some 20 roundings of 6e-8: weights, four stages, time weights, sums)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("im,vm", [((256, 256), (4, 4)), ((64, 48, 80), (4, 3, 5))])
@pytest.mark.parametrize("K,N", [(1, 2), (3, 4), (9, 4)])
def test_small_corner_weights(im, vm, K, N):
    from paper_1703_04446_gb300 import lgnk
    d = len(im)
    ratio = im[0] // vm[0]
    at = [ratio // 2 + ratio - 1] * d                 # offset 1 - 1 / (2 ratio) in cell (0, ..)
    f = (at[0] + 0.5) / ratio - 0.5
    assert 0.9 < f < 1.0
    ctx = lgnk.Context(lgnk.Problem(image_m=im, velocity_m=vm, time_nodes=K, rk4_steps=N, model="continuity"))
    T = torch.zeros(ctx.problem.image_shape, device="cuda")
    T[tuple(at)] = 1.0
    r = torch.zeros(ctx.problem.image_shape, device="cuda")
    for a in range(d):
        shape = [1] * d
        shape[d - 1 - a] = im[a]
        r += (a + 1) * torch.arange(im[a], device="cuda", dtype=torch.float32).reshape(shape)
    g = ctx.jtvp(torch.zeros(ctx.problem.velocity_shape, device="cuda"), T, r).cpu().numpy().astype(np.float64)
    ctx.close()
    g = g.sum(0)                                      # over the time nodes
    for a in range(d):
        total = g[a].sum()
        assert abs(total) > 0
        for c in range(1 << d):
            bits = [(c >> b) & 1 for b in range(d)]
            w = np.prod([f if b else 1.0 - f for b in bits])
            assert abs(g[a][tuple(reversed(bits))] / total - w) <= 2e-6 * w, (a, bits)
