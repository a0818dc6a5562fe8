"""The spectral preconditioner's transforms by halves (even and odd modes) against
the oracle, at the sizes where their indexing changes: axes of one to five cells,
odd lengths with an unpaired middle, lengths that are not multiples of the 4 x 4 or
4 x 8 register blocks, the largest half-table axis (128) and one past it, planes
with 4 and with 8 lines per thread, and a ragged last tile of lines.

Tolerance: the parity tests' 1e-5 (FP32 sums of at most 128 terms per axis and
direction, about 1e-6 relative in all)."""
import numpy as np
import pytest
import torch

from oracle import lagrangian as L
from oracle.objective import Problem as OProblem
from oracle.solver import apply_preconditioner
from tests._cases import rel

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 3), (5, 1), (3, 7), (64, 64), (65, 33), (96, 128), (128, 127), (129, 12), (12, 129),
         (1, 1, 1), (3, 2, 1), (1, 5, 3), (7, 4, 5), (33, 31, 17), (64, 64, 2), (96, 112, 20), (128, 128, 3),
         (30, 22, 128), (127, 9, 64), (129, 5, 6), (10, 131, 8), (10, 8, 130)]


@pytest.mark.parametrize("vm", SIZES)
@pytest.mark.parametrize("reg,gamma", [("diffusion", 0.0), ("curvature", 1e-3)])
def test_preconditioner_by_halves(vm, reg, gamma):
    from paper_1703_04446_gb300 import lgnk
    d, K = len(vm), 2
    if gamma == 0.0 and max(vm) == 1:
        gamma = 1e-3                       # a single cell has the constant mode only
    im = tuple(2 * a for a in vm)
    op = OProblem(L.Grid(im), L.Grid(vm), K=K, N=2, reg=reg, alpha=1e-2, gamma=gamma)
    ctx = lgnk.Context(lgnk.Problem(image_m=im, velocity_m=vm, time_nodes=K, rk4_steps=2, regularizer=reg, alpha=1e-2,
                                    gamma=gamma))
    r = np.random.default_rng(7).normal(size=(K, d) + tuple(reversed(vm))).astype(np.float32)
    got = ctx.precond(torch.from_numpy(r).cuda()).cpu().numpy().astype(np.float64)
    ctx.close()
    assert rel(got, apply_preconditioner(op, r.astype(np.float64))) <= 1e-5
