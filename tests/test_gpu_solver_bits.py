"""The rounding of the solver's sums stays what it was.

The second Gauss-Newton step takes grad T, which jumps at image nodes, at end
points of the first step's velocity: a change of that velocity by a rounding
can move a voxel's row of J by O(1), so the sums that make a solve's iterates
(the rows of J, the preconditioner in PCG) keep their order.  The checksums in
``golden/solver_bits.json`` are of outputs without order-dependent additions:
J dv has none, and with the velocity on the image's own grid and v = 0 every
voxel adds to one node only, so v after one step has none either.

``python -m tests.test_gpu_solver_bits`` prints the checksums of the built
library."""
import json
import os
import zlib

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "solver_bits.json")

# J dv of assembled rows: image cells, velocity cells, time nodes, RK4 steps
ROWS = [((20, 18, 16), (10, 9, 8), 1, 4), ((16, 16, 16), (16, 16, 16), 1, 8), ((14, 16, 18), (7, 8, 9), 3, 4),
        ((40, 36), (20, 18), 1, 4), ((32, 32), (32, 32), 2, 8)]
# one step of a 3D solve: cells of both grids; planes of at most and of more than 64 x 64
# cells, a last axis of more than 64 and of more than 128 cells, odd sizes, small axes
STEPS = [(16, 12, 10), (64, 64, 8), (13, 9, 11), (72, 10, 12), (8, 9, 72), (6, 5, 130), (130, 4, 6), (4, 67, 5),
         (3, 2, 1), (48, 40, 56)]


def _values(shape, seed, scale):
    """Multiples of scale / 128 in (-scale, scale), the same on every machine."""
    n = int(np.prod(shape))
    x = (np.arange(n, dtype=np.uint64) + np.uint64(977 * seed + 1)) * np.uint64(0x9E3779B97F4A7C15)
    x ^= x >> np.uint64(29)
    x *= np.uint64(0xBF58476D1CE4E5B9)
    i = (x >> np.uint64(56)).astype(np.int64) - 128
    return torch.from_numpy((i * (scale / 128.0)).astype(np.float32).reshape(shape)).cuda()


def _crc(t):
    return zlib.crc32(t.detach().cpu().numpy().tobytes())


def _rows(im, vm, K, N):
    from paper_1703_04446_gb300 import lgnk
    ctx = lgnk.Context(lgnk.Problem(image_m=im, velocity_m=vm, time_nodes=K, rk4_steps=N))
    v = _values(ctx.problem.velocity_shape, 1, 0.25)
    T = _values(ctx.problem.image_shape, 2, 1.0)
    ctx.assemble(v, T)
    du = ctx.jvp_assembled(_values(ctx.problem.velocity_shape, 3, 0.25))
    out = _crc(du)
    ctx.close()
    return out


def _step(m):
    from paper_1703_04446_gb300 import lgnk
    ctx = lgnk.Context(lgnk.Problem(image_m=m, velocity_m=m, time_nodes=1, rk4_steps=2, alpha=2.0 ** -10))
    T, R = _values(ctx.problem.image_shape, 4, 1.0), _values(ctx.problem.image_shape, 5, 1.0)
    v, rep = ctx.solve(T, R, None, max_gn=1, max_pcg=4, pcg_rtol=1e-9, gn_grad_rtol=1e-9)
    assert rep["hessvecs"] == 4
    out = _crc(v)
    ctx.close()
    return out


def _name(*a):
    return " ".join("x".join(map(str, x)) if isinstance(x, tuple) else str(x) for x in a)


def _golden():
    with open(GOLDEN) as f:
        return json.load(f)


@pytest.mark.parametrize("im,vm,K,N", ROWS)
def test_rows_keep_their_rounding(im, vm, K, N):
    assert _rows(im, vm, K, N) == _golden()["rows"][_name(im, vm, K, N)]


@pytest.mark.parametrize("m", STEPS)
def test_first_step_keeps_its_rounding(m):
    assert _step(m) == _golden()["steps"][_name(m)]


if __name__ == "__main__":
    print(json.dumps({"rows": {_name(*a): _rows(*a) for a in ROWS}, "steps": {_name(m): _step(m) for m in STEPS}},
                     indent=1))
