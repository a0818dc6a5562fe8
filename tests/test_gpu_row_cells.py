"""The Gauss-Newton product by rows (3D, stationary velocity, N >= 4) falls back to
tangent sweeps when the characteristics cross many velocity cells: both sides of
that rule against the FP64 oracle, and the cost that the rule keeps out.

Tolerance: the parity tests' 1e-5."""
import numpy as np
import pytest
import torch

from oracle import lagrangian as L
from oracle.objective import Problem as OProblem, hessvec
from paper_1703_04446_gb300 import synth
from tests._cases import rel

pytestmark = pytest.mark.gpu


def _mean_faces(v, vm):
    """The kernel's sample: cell faces crossed at the speed of 64 nodes."""
    t = np.arange(64, dtype=np.float32) + np.float32(0.5)
    idx = []
    for a, s in enumerate((0.8191725, 0.6710436, 0.5497005)):
        x = t * np.float32(s)
        idx.append(np.minimum(((x - np.floor(x)) * vm[a]).astype(int), vm[a] - 1))
    s = v[0][:, idx[2], idx[1], idx[0]]
    return float(sum(np.abs(s[a]) * vm[a] for a in range(3)).mean())


@pytest.mark.parametrize("vm,N,cells,many", [((16, 18, 20), 4, 0.5, False), ((16, 18, 20), 4, 6.0, True),
                                             ((8, 9, 10), 4, 3.0, False), ((16, 18, 20), 8, 1.5, False),
                                             ((16, 18, 20), 8, 8.0, True), ((16, 18, 20), 16, 12.0, True)])
def test_product_on_both_sides_of_the_rule(vm, N, cells, many):
    from paper_1703_04446_gb300 import lgnk
    im = (16, 18, 20)
    lo, hi = (0.0,) * 3, (1.0,) * 3
    ig, vg = synth.GridSpec(im, lo, hi), synth.GridSpec(vm, lo, hi)
    coords = synth.centres(ig)
    T = synth.gaussian_blobs(coords, [(1.0, 0.2, (0.45,) * 3), (0.6, 0.12, (0.6,) * 3)]).astype(np.float32)
    v = np.ascontiguousarray(synth.random_velocity(vg, 1, cells / 16, 4, n_modes=1), dtype=np.float32)
    dv = np.ascontiguousarray(synth.random_velocity(vg, 1, 2.0 / 16, 5), dtype=np.float32)
    assert (_mean_faces(v, vm) > min(0.12 * N, 1.1)) == many
    op = OProblem(L.Grid(im, lo, hi), L.Grid(vm, lo, hi), K=1, N=N, model="transport", reg="diffusion", alpha=1e-3,
                  gamma=1e-3)
    ctx = lgnk.Context(lgnk.Problem(image_m=im, velocity_m=vm, time_nodes=1, rk4_steps=N, alpha=1e-3, gamma=1e-3))
    got = ctx.hessvec(*(torch.from_numpy(a).cuda() for a in (v, T, dv))).cpu().numpy().astype(np.float64)
    ctx.close()
    assert rel(got, hessvec(op, *(a.astype(np.float64) for a in (v, T, dv)))) <= 1e-5


@pytest.mark.parametrize("N", [4, 8])
def test_product_over_many_cells_costs_less_than_its_parts(N):
    """J^T h^d J dv traces once where J dv and J^T r trace twice (by rows it took 1.05 to
    1.12 of the two at these sizes, by tangents 0.83)."""
    from paper_1703_04446_gb300 import lgnk
    m = (96, 96, 96)
    ctx = lgnk.Context(lgnk.Problem(image_m=m, velocity_m=m, time_nodes=1, rk4_steps=N))
    g = synth.GridSpec(m, (0.0,) * 3, (1.0,) * 3)
    v = torch.from_numpy(np.ascontiguousarray(synth.random_velocity(g, 1, 25.0 / 96, 4), dtype=np.float32)).cuda()
    T, r = torch.rand(ctx.problem.image_shape, device="cuda"), torch.rand(ctx.problem.image_shape, device="cuda")
    dv = torch.rand(ctx.problem.velocity_shape, device="cuda")

    def time(fn):
        best = []
        for _ in range(12):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(5):
                fn()
            e[1].record()
            torch.cuda.synchronize()
            best.append(e[0].elapsed_time(e[1]))
        return min(best[2:])

    parts = time(lambda: ctx.jvp(v, T, dv)) + time(lambda: ctx.jtvp(v, T, r))
    whole = time(lambda: ctx.hessvec(v, T, dv))
    ctx.close()
    assert whole < parts
