"""The tracing kernels' choices by time nodes K, steps N and displacement,
against the FP64 oracle: gradients accumulated per stage time (K - 1 > N), on
the time nodes (K - 1 <= N, with equality at the boundary of the rule), and
Gauss-Newton rows with more blocks than a thread keeps.

Tolerance: the parity tests' 1e-5 (FP32 tracing against FP64: rounding of about
6e-8 a stage, amplified 1e2 by the 4 N stages and the corner sums)."""
import functools

import numpy as np
import pytest
import torch

from oracle import lagrangian as L
from oracle.objective import Problem as OProblem, gradient, hessvec
from paper_1703_04446_gb300 import synth
from tests._cases import rel

pytestmark = pytest.mark.gpu
TOL = 1e-5

# name: (image m, velocity m, K, N, model, displacement in image cells)
CASES = {
    "3d_transport_K5_N2": ((20, 18, 17), (10, 9, 9), 5, 2, "transport", 2.5),
    "3d_mass_K5_N2": ((20, 18, 17), (10, 9, 9), 5, 2, "continuity", 2.0),
    "3d_transport_K4_N3": ((20, 18, 17), (10, 9, 9), 4, 3, "transport", 2.5),
    "3d_mass_K4_N3": ((20, 18, 17), (10, 9, 9), 4, 3, "continuity", 2.0),
    "3d_mass_K3_N8": ((16, 20, 12), (8, 10, 6), 3, 8, "continuity", 2.0),
    "3d_transport_K1_far": ((24, 22, 20), (24, 22, 20), 1, 16, "transport", 8.0),
    "3d_transport_K9_far": ((24, 22, 20), (24, 22, 20), 9, 8, "transport", 6.0),
    "2d_transport_K6_N2": ((37, 29), (19, 15), 6, 2, "transport", 3.0),
    "2d_mass_K6_N2": ((37, 29), (19, 15), 6, 2, "continuity", 3.0),
    "2d_transport_K6_N5": ((37, 29), (19, 15), 6, 5, "transport", 3.0),
    "2d_mass_K6_N5": ((37, 29), (19, 15), 6, 5, "continuity", 3.0),
    "2d_transport_K1_far": ((48, 40), (48, 40), 1, 16, "transport", 12.0),
    "2d_transport_K3_far": ((48, 40), (48, 40), 3, 16, "transport", 12.0),
}


@functools.lru_cache(maxsize=None)
def _case(name):
    im, vm, K, N, model, amp = CASES[name]
    d = len(im)
    lo, hi = (0.0,) * d, (1.0,) * d
    ig, vg = synth.GridSpec(im, lo, hi), synth.GridSpec(vm, lo, hi)
    rng = np.random.default_rng(3)
    coords = synth.centres(ig)
    blobs = [(1.0, 0.2, (0.45,) * d), (0.6, 0.12, (0.6,) * d)]
    T, R = synth.gaussian_blobs(coords, blobs), synth.gaussian_blobs([c - 0.03 for c in coords], blobs)
    h = min(ig.h)
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    a = dict(T=f32(T), R=f32(R), v=f32(synth.random_velocity(vg, K, amp * h, 4, n_modes=1)),
             dv=f32(synth.random_velocity(vg, K, 2.0 * h, 5)),
             r=f32(synth.gaussian_blobs(coords, [(1.0, 0.15, (0.5,) * d)]) + 0.1 * rng.normal(size=T.shape)))
    op = OProblem(L.Grid(im, lo, hi), L.Grid(vm, lo, hi), K=K, N=N, model=model, reg="diffusion", alpha=1e-3,
                  gamma=1e-3)
    gp = dict(image_m=im, velocity_m=vm, time_nodes=K, rk4_steps=N, model=model, alpha=1e-3, gamma=1e-3)
    return op, gp, a


@pytest.mark.parametrize("name", list(CASES))
def test_products_match_the_oracle(name):
    from paper_1703_04446_gb300 import lgnk
    op, gp, a = _case(name)
    f64 = {k: v.astype(np.float64) for k, v in a.items()}
    t = {k: torch.from_numpy(v).cuda() for k, v in a.items()}
    ctx = lgnk.Context(lgnk.Problem(**gp))
    args = (op.vgrid, f64["T"], op.igrid, op.N)
    u1, y = L.final_state(op.model, f64["v"], *args, op.delta)
    if name.endswith("_far"):      # rows with more blocks than a thread keeps (6; 12 on the time nodes)
        idx = np.stack([c.reshape(-1) for c in synth.centres(synth.GridSpec(gp["image_m"], op.igrid.lo, op.igrid.hi))])
        cells = np.abs(np.floor(y.reshape(idx.shape) * np.array(gp["velocity_m"])[:, None] - 0.5)
                       - np.floor(idx * np.array(gp["velocity_m"])[:, None] - 0.5)).sum(0)
        # a new cell ends one block, or with time nodes the blocks of both nodes
        blocks = cells.max() + 1 if gp["time_nodes"] == 1 else 2 * cells.max() + gp["time_nodes"]
        assert blocks > (8 if gp["time_nodes"] == 1 else 14)
    np_ = lambda x: x.detach().cpu().numpy().astype(np.float64)
    err = {
        "u1": rel(np_(ctx.forward(t["v"], t["T"])), u1),
        "jvp": rel(np_(ctx.jvp(t["v"], t["T"], t["dv"])), L.jvp(op.model, f64["v"], *args, f64["dv"], op.delta)),
        "jtvp": rel(np_(ctx.jtvp(t["v"], t["T"], t["r"])), L.jtvp(op.model, f64["v"], *args, f64["r"], op.delta)),
        "hess": rel(np_(ctx.hessvec(t["v"], t["T"], t["dv"])), hessvec(op, f64["v"], f64["T"], f64["dv"])),
        "grad": rel(np_(ctx.objective(t["v"], t["T"], t["R"], grad=True)[3]),
                    gradient(op, f64["v"], f64["T"], f64["R"])),
    }
    ctx.close()
    assert max(err.values()) <= TOL, err
