"""The work that a user of this package has it do, as cases to be timed.

A case is one pass through public entry points (``Context.forward``,
``hessvec``, ``objective``, ``assemble`` with the assembled products,
``precond``, ``solve``, the autograd wrapper, and the warm-start network), on
seeded inputs shaped like the registration problems of ``synth.WORKLOADS``.

``listed()`` names the cases, ``draw()`` gives more of the same ranges,
``prepare()`` makes what a program has in hand before the call (inputs,
context, network), ``run()`` makes one pass, ``work()`` counts what the pass
cannot do without, and ``exact()`` evaluates it in 64 bits with plain torch.
"""
import math
import random

import torch
import torch.nn.functional as F

from paper_1703_04446_gb300 import lgnk

PAD = 2          # zero nodes around the grids of the 64-bit evaluation
CHUNK = 1 << 20  # particles traced together in 64 bits


def _m(text):
    return tuple(int(a) for a in text.split("x"))


def _text(m):
    return "x".join(str(a) for a in m)


def _half(m):
    return tuple((a + 1) // 2 for a in m)


def _problem(kind, image, K, N, model="transport", reg="diffusion", alpha=1e-2, disp=8.0, gamma=0.0,
             **more):
    """A registration problem: images of `image` cells, a velocity of half as
    many per axis on K time nodes, N RK4 steps, displacements of `disp` cells."""
    return dict(kind=kind, image=_text(image), velocity=_text(_half(image)), K=K, N=N, model=model, reg=reg,
                alpha=alpha, gamma=gamma, disp=disp, **more)


def listed():
    return [
        # the smallest call: the final state of a 64^2 pair (launch latency)
        dict(name="forward_2d_64", **_problem("forward", (64, 64), 1, 4, disp=6.0)),
        # a Gauss-Newton product of the mass-preserving 2D workload (256^2, 5 time nodes, elastic)
        dict(name="hessvec_2d_mass_256", **_problem("hessvec", (256, 256), 5, 16, "continuity", "elastic", 1e-3, 12.0)),
        # the matrix-free Gauss-Newton product of the 3D workload, the benchmark's step
        dict(name="hessvec_3d_128", **_problem("hessvec", (128, 128, 128), 1, 8)),
        # objective and gradient on a volume of odd sizes (one evaluation of a matrix-free Gauss-Newton step)
        dict(name="objective_3d_odd", **_problem("objective", (109, 131, 93), 1, 8, disp=6.0)),
        # the work of one Gauss-Newton step of the default solver at 128^3: J assembled, then the PCG's products
        dict(name="assembled_3d_128", **_problem("assembled", (128, 128, 128), 1, 8, products=8)),
        # non-stationary transport at the sizes of the paper's 3D experiment (two time nodes, curvature)
        dict(name="hessvec_3d_K2", **_problem("hessvec", (128, 150, 128), 2, 5, "transport", "curvature", 1e-5, 6.0)),
        # the largest call: the mass-preserving Gauss-Newton product at brain scale (9 time nodes)
        dict(name="hessvec_3d_mass_brain",
             **_problem("hessvec", (192, 224, 160), 9, 16, "continuity", "diffusion", 1e-3, 6.0)),
        # the spectral preconditioner on the brain-scale velocity (axes beyond the 64-cell planes)
        dict(name="precond_3d_brain",
             **_problem("precond", (192, 224, 160), 9, 16, "continuity", "diffusion", 1e-3, 6.0)),
        # one prediction of the learned warm start (what a warm-started solve waits for)
        dict(name="predict_128_b1", kind="predict", m=128, channels=32, batch=1),
        # one training step of the warm start at its batch size, with its gradients and updated weights
        dict(name="train_128_b32", kind="train", m=128, channels=32, batch=32),
        # the first steps of a 2D solve of the warm start's target generation: many small kernels and host waits
        dict(name="solve_2d_128",
             **_problem("solve", (128, 128), 1, 4, alpha=1e-3, disp=8.0, gamma=1e-3, max_gn=2, max_pcg=10)),
        # the first Gauss-Newton steps of a 3D solve from zero with a fixed count of PCG iterations
        dict(name="solve_3d_128", **_problem("solve", (128, 128, 128), 1, 8, max_gn=2, max_pcg=8)),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    kind = rng.choice(["forward", "hessvec", "hessvec", "objective", "assembled", "precond", "autograd", "predict",
                       "train", "solve"])
    if kind in ("predict", "train"):
        m = 8 * rng.randint(4, 20)
        batch = max(1, min(int(_log(rng, 1, 48)), int(32 * 128 * 128 / (m * m))))
        return dict(kind=kind, m=m, channels=rng.choice([8, 16, 24, 32]), batch=batch)
    d = rng.choice([2, 3, 3])
    side = _log(rng, 24, 400) if d == 2 else _log(rng, 20, 150)
    image = tuple(max(9, int(side * rng.uniform(0.75, 1.2))) for _ in range(d))
    mass = kind not in ("assembled", "solve") and rng.random() < 0.4
    K = 1 if kind in ("assembled", "solve") else rng.choice([1, 1, 2, 3, 5, 9])
    N = rng.choice([2, 4, 5, 8]) if kind in ("assembled", "solve") or d == 3 else rng.choice([2, 4, 5, 8, 16])
    more = {}
    if kind == "assembled":
        more = dict(products=rng.randint(4, 12))
    if kind == "solve":
        more = dict(max_gn=rng.randint(1, 2), max_pcg=rng.randint(4, 8))
    reg = "diffusion" if kind == "solve" else rng.choice(["diffusion", "diffusion", "curvature", "elastic"])
    alpha = rng.choice([1e-2, 1e-3]) * (1e-3 if reg == "curvature" else 1.0)
    case = _problem(kind, image, K, N, "continuity" if mass else "transport", reg, alpha,
                    disp=min(6.0, 0.05 * side + 1.0), **more)
    case["gamma"] = (1e-3 if d == 2 else 0.0) if kind == "solve" else rng.choice([0.0, 1e-3])
    return case


# ------------------------------------------------------------------ inputs --


def _axes(m, dtype=torch.float32):
    """Box-normalised cell-centre coordinates (x, y[, z]) that broadcast to the array shape (z, y, x)."""
    d = len(m)
    out = []
    for a in range(d):
        x = (torch.arange(m[a], device="cuda", dtype=dtype) + 0.5) / m[a]
        out.append(x.reshape([-1 if d - 1 - i == a else 1 for i in range(d)]))
    return out


def _smooth(m, rng, amplitude):
    """A smooth vector field (d, *grid) of four Fourier modes that vanishes on the box's boundary."""
    d = len(m)
    ax = _axes(m)
    window = 1.0
    for x in ax:
        window = window * torch.sin(math.pi * x) ** 2
    out = [0.0] * d
    for _ in range(4):
        k = [rng.randint(1, 3) for _ in range(d)]
        phase = rng.uniform(0.0, 2.0 * math.pi)
        s = torch.sin(2.0 * math.pi * sum(kk * x for kk, x in zip(k, ax)) + phase)
        for c in range(d):
            out[c] = out[c] + rng.gauss(0.0, 1.0) * s
    f = torch.stack([o * window for o in out])
    return f * (amplitude / f.square().sum(0).sqrt().max().clamp_min(1e-12))


def _velocity(m, K, rng, amplitude):
    a, b = _smooth(m, rng, amplitude), _smooth(m, rng, amplitude)
    w = [j / (K - 1) if K > 1 else 0.0 for j in range(K)]
    return torch.stack([(1.0 - s) * a + s * b for s in w]).contiguous()


def _blobs(coords, params):
    out = 0.0
    for amp, sigma, centre in params:
        out = out + amp * torch.exp(-sum((x - c) ** 2 for x, c in zip(coords, centre)) / (2.0 * sigma * sigma))
    return out


def _phantom(coords, params):
    """Nested tanh-edged ellipsoids with an intensity ramp."""
    centre, levels = params
    out = 0.0
    for radii, inten in levels:
        r = sum(((x - c) / a) ** 2 for x, c, a in zip(coords, centre, radii)).sqrt()
        out = out + inten * (1.0 + 0.3 * (coords[0] - centre[0])) * 0.5 * (1.0 - torch.tanh((r - 1.0) / 0.06))
    return out


def _images(m, rng, gen, mass, disp_cells):
    """Template and reference: blobs (2D) or a noisy phantom (3D), the reference the analytic template displaced."""
    d = len(m)
    ax = _axes(m)
    s = _smooth(m, rng, disp_cells / max(m))
    moved = [x - s[a] for a, x in enumerate(ax)]
    if d == 2:
        params = [(rng.uniform(0.4, 1.0), rng.uniform(0.05, 0.12), [rng.uniform(0.2, 0.8) for _ in range(d)])
                  for _ in range(8)]
        T, R = _blobs(ax, params), _blobs(moved, params)
    else:
        centre = [0.5 + rng.uniform(-0.03, 0.03) for _ in range(d)]
        params = (centre, [([scale * rng.uniform(0.85, 1.15) for _ in range(d)], inten)
                           for scale, inten in ((0.38, 0.5), (0.26, 0.3), (0.14, 0.2))])
        T, R = _phantom(ax, params), _phantom(moved, params)
    if mass:
        T, R = T / T.mean(), R / R.mean()
    else:
        T = T + 0.01 * torch.randn(T.shape, device="cuda", generator=gen)
        R = R + 0.01 * torch.randn(R.shape, device="cuda", generator=gen)
    return T.contiguous(), R.contiguous()


def _inputs(case, seed):
    rng = random.Random(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["kind"] in ("predict", "train"):
        return _net_inputs(case, rng, gen)
    im, vm = _m(case["image"]), _m(case["velocity"])
    K, amp = case["K"], case["disp"] / max(im)
    if case["kind"] == "precond":   # a residual of the velocity's shape
        return {"r": _velocity(vm, K, rng, 1e-3) + 1e-4 * torch.randn((K, len(vm)) + vm[::-1], device="cuda",
                                                                     generator=gen)}
    T, R = _images(im, rng, gen, case["model"] == "continuity", case["disp"])
    if case["kind"] == "solve":
        return {"T": T, "R": R}
    out = {"T": T, "R": R, "v": _velocity(vm, K, rng, amp)}
    if case["kind"] in ("hessvec", "assembled"):    # PCG directions: smooth (preconditioned)
        n = case.get("products", 1)
        out["dv"] = [_velocity(vm, K, rng, 0.5 * amp) for _ in range(n)]
    if case["kind"] == "autograd":
        out["r"] = torch.randn(T.shape, device="cuda", generator=gen)
    return out


def _layers(c):
    """(input channels, output channels, stride, input upsampled) of the warm-start network."""
    return [(2, c, 1, 0), (c, 2 * c, 2, 0), (2 * c, 4 * c, 2, 0), (4 * c, 8 * c, 2, 0), (8 * c, 4 * c, 1, 1),
            (4 * c, 2 * c, 1, 1), (2 * c, 2, 1, 0)]


SCALE = 0.05    # the network's output scale
LR = 1e-5       # the end of the training's learning-rate schedule


def _net_inputs(case, rng, gen):
    m, c, B = case["m"], case["channels"], case["batch"]
    p = []
    for ci, co, _, _ in _layers(c):     # He-normal weights, small biases
        p.append(torch.randn(co * ci * 9, device="cuda", generator=gen) * math.sqrt(2.0 / (9 * ci)))
        p.append(0.01 * torch.randn(co, device="cuda", generator=gen))
    pairs = [_images((m, m), rng, gen, False, 0.06 * m) for _ in range(B)]
    target = torch.stack([_smooth((m // 2, m // 2), rng, 0.06) for _ in range(B)])
    return {"p": torch.cat(p), "T": torch.stack([a for a, _ in pairs]), "R": torch.stack([b for _, b in pairs]),
            "target": target.contiguous()}


def _lgnk_problem(case):
    return lgnk.Problem(image_m=_m(case["image"]), velocity_m=_m(case["velocity"]), time_nodes=case["K"],
                        rk4_steps=case["N"], model=case["model"], regularizer=case["reg"], alpha=case["alpha"],
                        gamma=case["gamma"])


def prepare(case, seed):
    state = _inputs(case, seed)
    state["case"] = case
    if case["kind"] in ("predict", "train"):
        net = lgnk.WarmStart(case["m"], case["channels"], case["batch"], SCALE)
        net.set_params(state.pop("p"))
        state["net"] = net
    else:
        state["ctx"] = lgnk.Context(_lgnk_problem(case))
    if case["kind"] == "autograd":
        state["v"].requires_grad_(True)
    return state


# -------------------------------------------------------------------- run --


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "predict":
        return s["net"].predict(s["T"], s["R"])
    if kind == "train":
        s["net"].train_step(s["T"], s["R"], s["target"], LR, return_loss=False)
        return {"grads": s["net"].grads(), "params": s["net"].params()}
    ctx = s["ctx"]
    if kind == "forward":
        return ctx.forward(s["v"], s["T"])
    if kind == "hessvec":
        return ctx.hessvec(s["v"], s["T"], s["dv"][0])
    if kind == "objective":
        J, D, S, g = ctx.objective(s["v"], s["T"], s["R"], grad=True)
        return {"J": J, "D": D, "S": S, "grad": g}
    if kind == "assembled":
        ctx.assemble(s["v"], s["T"])
        return [ctx.hessvec_assembled(dv) for dv in s["dv"]]
    if kind == "precond":
        return ctx.precond(s["r"])
    if kind == "autograd":
        u1 = lgnk.lagrangian_forward(ctx, s["v"], s["T"])
        (g,) = torch.autograd.grad(u1, s["v"], s["r"])
        return {"u1": u1.detach(), "grad": g}
    v, rep = ctx.solve(s["T"], s["R"], None, max_gn=case["max_gn"], max_pcg=case["max_pcg"], pcg_rtol=1e-9,
                       gn_grad_rtol=1e-9)
    return {"v": v, "J": rep["J"], "J0": rep["J0"]}


# ------------------------------------------------------------------- work --


def work(case):
    """Bytes: each input read and each output written once.  Operations: the
    RK4 stages' multilinear values (and, with derivatives, their gradients and
    the transposed accumulation) per particle and step, the network's
    convolutions, or the preconditioner's two transforms per axis."""
    if case["kind"] in ("predict", "train"):
        m, B = case["m"], case["batch"]
        h, flops, params = m, 0.0, 0
        for ci, co, s, up in _layers(case["channels"]):
            ho = 2 * h if up else h // s
            flops += 2.0 * 9 * ci * co * ho * ho * B
            params += 9 * ci * co + co
            h = ho
        data = 4.0 * B * (2 * m * m + 2 * (m // 2) ** 2)
        return {"bytes": data + (4.0 * params if case["kind"] == "predict" else 28.0 * params),
                "flops": flops if case["kind"] == "predict" else 3.0 * flops}
    im, vm = _m(case["image"]), _m(case["velocity"])
    d, M = len(im), float(math.prod(im))
    n = float(math.prod(vm)) * d * case["K"]
    kind = case["kind"]
    if kind == "precond":
        return {"bytes": 8.0 * n, "flops": 4.0 * n * sum(vm)}
    steps = M * case["N"]
    value, tangent, adjoint = (210.0, 630.0, 454.0) if d == 3 else (90.0, 240.0, 190.0)
    if kind == "forward":
        return {"bytes": 4.0 * (n + 2 * M), "flops": value * steps}
    if kind == "hessvec":
        return {"bytes": 4.0 * (3 * n + M), "flops": (tangent + adjoint) * steps}
    if kind == "objective":
        return {"bytes": 4.0 * (2 * n + 2 * M), "flops": (value + adjoint) * steps}
    if kind == "autograd":
        return {"bytes": 4.0 * (3 * n + 3 * M), "flops": (2 * value + adjoint) * steps}
    row = (2 ** d) * d      # one block of a row of J: written once, read once per product
    if kind == "assembled":
        k = case["products"]
        return {"bytes": 4.0 * (n + M + (k + 1) * row * M + 2 * k * n),
                "flops": (value + adjoint) * steps + 4.0 * k * row * M}
    g, p = case["max_gn"], case["max_gn"] * case["max_pcg"]
    return {"bytes": 4.0 * ((g + 1 + p) * row * M + p * 8 * n),
            "flops": (g + 1) * (value + adjoint) * steps + p * (4.0 * row * M + 4.0 * n * sum(vm))}


# ------------------------------------------------------------------ exact --


class _Tracer:
    """RK4 characteristics, their tangents and adjoints in 64 bits (plain torch).

    Positions are displacements from the particle's start, whose index on
    either grid is exact, so that a particle which barely moves keeps the side
    of a cell face it moved to."""

    def __init__(self, case, v, dvs=()):
        self.im, self.vm = _m(case["image"]), _m(case["velocity"])
        self.d, self.K, self.N = len(self.im), case["K"], case["N"]
        self.transport = case["model"] == "transport"
        self.dt = (-1.0 if self.transport else 1.0) / self.N
        times = [min(1.0, max(0.0, (1.0 if self.transport else 0.0) + 0.5 * m * self.dt))
                 for m in range(2 * self.N + 1)]
        self.th = []
        for t in times:
            s = t * (self.K - 1)
            j = max(0, min(int(math.floor(s)), self.K - 2))
            self.th.append((j, s - j))
        self.v = self._pack(v)
        self.dv = [self._pack(x) for x in dvs]
        self.G = None

    def _pack(self, v):
        """[K][padded node][d]"""
        x = F.pad(v.double(), (PAD, PAD) * self.d)
        return x.reshape(self.K, self.d, -1).transpose(1, 2).contiguous()

    def _slice(self, table, m):
        if self.K == 1:
            return table[0]
        j, th = self.th[m]
        return table[j] if th == 0.0 else (1.0 - th) * table[j] + th * table[j + 1]

    @staticmethod
    def _pads(m):
        return [a + 2 * PAD for a in m]

    def locate(self, m, start, u, h):
        """(index of the lower corner in the padded grid, offsets) of the point at displacement u."""
        mp = self._pads(m)
        base, f = 0, []
        step = 1
        for a in range(self.d):
            t = (start[a] + u[a] / h[a]).clamp(-float(PAD), m[a] + 0.5)
            lo = torch.floor(t)
            f.append(t - lo)
            base = base + (lo.long() + PAD) * step
            step *= mp[a]
        return base, f

    def offsets(self, m):
        mp = self._pads(m)
        return [(c & 1) + ((c >> 1) & 1) * mp[0] + ((c >> 2) & 1 if self.d == 3 else 0) * mp[0] * mp[1]
                for c in range(1 << self.d)]

    def weights(self, f):
        out = []
        for c in range(1 << self.d):
            w = 1.0
            for a in range(self.d):
                w = w * (f[a] if (c >> a) & 1 else 1.0 - f[a])
            out.append(w)
        return out

    def dweights(self, f, h):
        """[axis][corner]"""
        out = []
        for b in range(self.d):
            row = []
            for c in range(1 << self.d):
                w = (1.0 if (c >> b) & 1 else -1.0) / h[b]
                for a in range(self.d):
                    if a != b:
                        w = w * (f[a] if (c >> a) & 1 else 1.0 - f[a])
                row.append(w)
            out.append(row)
        return out

    def starts(self, lo, hi):
        """Image indices of particles lo..hi-1 and their continuous indices on the velocity grid."""
        i = torch.arange(lo, hi, device="cuda")
        idx, on_v = [], []
        for a in range(self.d):
            x = i % self.im[a]
            i = i // self.im[a]
            idx.append(x.double())
            on_v.append((x.double() + 0.5) * (self.vm[a] / self.im[a]) - 0.5)
        return idx, on_v

    def trace(self, lo, hi, keep=False):
        """End displacements, their tangents along each dv, and (keep) the stages' (slice, cell, offsets)."""
        d, dt = self.d, self.dt
        hv = [1.0 / a for a in self.vm]
        off = self.offsets(self.vm)
        idx, on_v = self.starts(lo, hi)
        u = [torch.zeros(hi - lo, device="cuda", dtype=torch.float64) for _ in range(d)]
        dy = [[x.clone() for x in u] for _ in self.dv]
        stages = []
        for k in range(self.N):
            acc, dacc = [0.0] * d, [[0.0] * d for _ in self.dv]
            us, q = u, dy
            for st, (m, w, nxt) in enumerate(((2 * k, 1.0, 0.5), (2 * k + 1, 2.0, 0.5), (2 * k + 1, 2.0, 1.0),
                                              (2 * k + 2, 1.0, None))):
                base, f = self.locate(self.vm, on_v, us, hv)
                if keep:
                    stages.append((m, base, f))
                W = self.weights(f)
                V = self._slice(self.v, m)
                corner = [V[base + o] for o in off]
                val = sum(W[c][:, None] * corner[c] for c in range(len(off)))
                if self.dv:
                    J = [sum(x[:, None] * y for x, y in zip(row, corner)) for row in self.dweights(f, hv)]
                qn = []
                for e, table in enumerate(self.dv):
                    B = self._slice(table, m)
                    D = sum(W[c][:, None] * B[base + off[c]] for c in range(len(off)))
                    for a in range(d):
                        D = D + J[a] * q[e][a][:, None]
                    dacc[e] = [dacc[e][a] + w * D[:, a] for a in range(d)]
                    qn.append([dy[e][a] + nxt * dt * D[:, a] for a in range(d)] if nxt else None)
                acc = [acc[a] + w * val[:, a] for a in range(d)]
                if nxt:
                    us, q = [u[a] + nxt * dt * val[:, a] for a in range(d)], qn
            u = [u[a] + dt / 6.0 * acc[a] for a in range(d)]
            dy = [[x[a] + dt / 6.0 * g[a] for a in range(d)] for x, g in zip(dy, dacc)]
        return idx, u, dy, stages

    def image(self, padded, idx, u):
        """Value and gradient of the padded image at the end points, and the corners' weights there."""
        hi = [1.0 / a for a in self.im]
        base, f = self.locate(self.im, idx, u, hi)
        off = self.offsets(self.im)
        corner = [padded[base + o] for o in off]
        W, dW = self.weights(f), self.dweights(f, hi)
        return (sum(w * c for w, c in zip(W, corner)), [sum(w * c for w, c in zip(row, corner)) for row in dW],
                (base, off, W, dW))

    def adjoint(self, stages, lam):
        """Accumulates (d_v y)^T lam into the slices' gradients."""
        d, dt = self.d, self.dt
        hv = [1.0 / a for a in self.vm]
        off = self.offsets(self.vm)
        if self.G is None:
            nodes = math.prod(self._pads(self.vm))
            self.G = torch.zeros((2 * self.N + 1 if self.K > 1 else 1, nodes, d), device="cuda", dtype=torch.float64)

        def stage(s, mu):
            m, base, f = s
            V = self._slice(self.v, m)
            W, dW = self.weights(f), self.dweights(f, hv)
            M = torch.stack(mu, 1)
            dots = []
            G = self.G[m if self.K > 1 else 0]
            for c, o in enumerate(off):
                dots.append((V[base + o] * M).sum(1))
                G.index_add_(0, base + o, W[c][:, None] * M)
            return [sum(x * y for x, y in zip(row, dots)) for row in dW]

        for k in reversed(range(self.N)):
            s1, s2, s3, s4 = stages[4 * k:4 * k + 4]
            nu4 = stage(s4, [dt / 6.0 * x for x in lam])
            nu3 = stage(s3, [dt / 3.0 * x + dt * n for x, n in zip(lam, nu4)])
            nu2 = stage(s2, [dt / 3.0 * x + 0.5 * dt * n for x, n in zip(lam, nu3)])
            nu1 = stage(s1, [dt / 6.0 * x + 0.5 * dt * n for x, n in zip(lam, nu2)])
            lam = [x + a + b + c + e for x, a, b, c, e in zip(lam, nu1, nu2, nu3, nu4)]

    def gradient(self):
        """The slices' gradients on the time nodes, in the velocity's layout."""
        vm, d = self.vm, self.d
        out = torch.zeros((self.K, self.G.shape[1], d), device="cuda", dtype=torch.float64)
        if self.K == 1:
            out[0] = self.G[0]
        else:
            for m, (j, th) in enumerate(self.th):
                out[j] += (1.0 - th) * self.G[m]
                out[j + 1] += th * self.G[m]
        self.G = None
        g = out.transpose(1, 2).reshape((self.K, d) + tuple(a + 2 * PAD for a in reversed(vm)))
        inner = (slice(None), slice(None)) + (slice(PAD, -PAD),) * d
        return g[inner].contiguous()


def _laplacian(x, h):
    """B^T B of the trailing grid axes, Neumann ends; h in axis order (x first)."""
    out = torch.zeros_like(x)
    for a in range(len(h)):
        dim = x.dim() - 1 - a
        if x.shape[dim] > 1:
            df = torch.diff(x, dim=dim) / (h[a] * h[a])
            n = x.shape[dim]
            out.narrow(dim, 0, n - 1).sub_(df)
            out.narrow(dim, 1, n - 1).add_(df)
    return out


def _centred(x, h, dim, transpose=False):
    """Centred difference along dim with mirrored ends, or its transpose."""
    n = x.shape[dim]
    up = torch.cat([x.narrow(dim, 1, n - 1), x.narrow(dim, n - 1, 1)], dim)
    dn = torch.cat([x.narrow(dim, 0, 1), x.narrow(dim, 0, n - 1)], dim)
    if not transpose:
        return (up - dn) / (2.0 * h)
    out = torch.zeros_like(x)
    out.narrow(dim, 1, n - 1).add_(x.narrow(dim, 0, n - 1))
    out.narrow(dim, n - 1, 1).add_(x.narrow(dim, n - 1, 1))
    out.narrow(dim, 0, n - 1).sub_(x.narrow(dim, 1, n - 1))
    out.narrow(dim, 0, 1).sub_(x.narrow(dim, 0, 1))
    return out / (2.0 * h)


def _regularizer(case, x):
    """dt h_v^d A x (A the regularizer's operator; Lame constants mu = 1, lambda = 0)."""
    vm = _m(case["velocity"])
    h = [1.0 / a for a in vm]
    w = (1.0 if case["K"] == 1 else 1.0 / (case["K"] - 1)) * math.prod(h)
    A = _laplacian(x, h)
    if case["reg"] == "curvature":
        A = _laplacian(A, h)
    if case["reg"] == "elastic":
        d = len(vm)
        div = sum(_centred(x[:, c], h[c], x.dim() - 2 - c) for c in range(d))
        A = A + torch.stack([_centred(div, h[c], div.dim() - 1 - c, True) for c in range(d)], 1)
    return w * A


def _chunks(M):
    return [(a, min(M, a + CHUNK)) for a in range(0, M, CHUNK)]


def _pad_image(T, d):
    return F.pad(T.double(), (PAD, PAD) * d).reshape(-1)


def _splat(tr, case, per_corner):
    """The push-forward of per-particle corner masses; per_corner(lo, hi) gives (base, offsets, masses)."""
    padded = torch.zeros(math.prod(tr._pads(tr.im)), device="cuda", dtype=torch.float64)
    for lo, hi in _chunks(math.prod(tr.im)):
        base, off, mass = per_corner(lo, hi)
        for o, x in zip(off, mass):
            padded.index_add_(0, base + o, x)
    full = padded.reshape([a + 2 * PAD for a in reversed(tr.im)])
    return full[(slice(PAD, -PAD),) * tr.d].contiguous()


def _forward64(tr, case, T):
    flat = T.double().reshape(-1)
    if tr.transport:
        padded = _pad_image(T, tr.d)
        out = torch.empty_like(flat)
        for lo, hi in _chunks(flat.numel()):
            idx, u, _, _ = tr.trace(lo, hi)
            out[lo:hi] = tr.image(padded, idx, u)[0]
        return out.reshape(T.shape)
    zero = _pad_image(torch.zeros_like(T), tr.d)

    def corners(lo, hi):
        idx, u, _, _ = tr.trace(lo, hi)
        base, off, W, _ = tr.image(zero, idx, u)[2]
        return base, off, [w * flat[lo:hi] for w in W]
    return _splat(tr, case, corners)


def _jtvp64(tr, case, T, r):
    flat = T.double().reshape(-1)
    padded = _pad_image(T if tr.transport else r, tr.d)
    scale = r.double().reshape(-1) if tr.transport else flat
    for lo, hi in _chunks(flat.numel()):
        idx, u, _, stages = tr.trace(lo, hi, keep=True)
        grad = tr.image(padded, idx, u)[1]
        tr.adjoint(stages, [scale[lo:hi] * g for g in grad])
    return tr.gradient()


def _products64(tr, case, T):
    """J^T h^d J dv for every direction of the tracer."""
    flat = T.double().reshape(-1)
    cell = 1.0 / math.prod(tr.im)
    if tr.transport:
        padded = _pad_image(T, tr.d)
        du = [torch.empty_like(flat) for _ in tr.dv]
        for lo, hi in _chunks(flat.numel()):
            idx, u, dys, _ = tr.trace(lo, hi)
            grad = tr.image(padded, idx, u)[1]
            for out, dy in zip(du, dys):
                out[lo:hi] = sum(g * y for g, y in zip(grad, dy))
    else:
        zero = _pad_image(torch.zeros_like(T), tr.d)

        def corners(lo, hi):
            idx, u, dys, _ = tr.trace(lo, hi)
            base, off, _, dW = tr.image(zero, idx, u)[2]
            return base, off, [flat[lo:hi] * sum(dW[a][c] * dys[0][a] for a in range(tr.d)) for c in range(len(off))]
        du = [_splat(tr, case, corners)]
    tr.dv = []
    return [_jtvp64(tr, case, T, cell * x.reshape(T.shape)) for x in du]


def _precond64(case, r):
    vm = _m(case["velocity"])
    d = len(vm)
    x = r.double()
    mats, lam = [], 0.0
    for a in range(d):
        m = vm[a]
        k = torch.arange(m, device="cuda", dtype=torch.float64)
        C = torch.cos(math.pi * k[:, None] * (2.0 * k[None, :] + 1.0) / (2.0 * m)) * math.sqrt(2.0 / m)
        C[0] /= math.sqrt(2.0)
        mats.append(C)
        e = (2.0 - 2.0 * torch.cos(math.pi * k / m)) * (m * m)
        lam = lam + e.reshape([-1 if d - 1 - i == a else 1 for i in range(d)])
    if case["reg"] == "curvature":
        lam = lam * lam
    w = (1.0 if case["K"] == 1 else 1.0 / (case["K"] - 1)) / math.prod(vm)
    p = case["alpha"] * w * lam + case["gamma"]
    p = torch.where(p > 0.0, p, p[p > 0.0].min())
    for a in range(d):
        x = torch.movedim(torch.tensordot(x, mats[a], dims=([x.dim() - 1 - a], [1])), -1, x.dim() - 1 - a)
    x = x / p
    for a in range(d):
        x = torch.movedim(torch.tensordot(x, mats[a], dims=([x.dim() - 1 - a], [0])), -1, x.dim() - 1 - a)
    return x.contiguous()


def _net64(case, s):
    """The warm-start network (weights rounded to bfloat16) and, for a training step, its gradient and Adam step."""
    params = s["p"]
    used = params.clone()
    at, pieces = 0, []
    for ci, co, _, _ in _layers(case["channels"]):
        n = co * ci * 9
        used[at:at + n] = params[at:at + n].bfloat16().float()
        pieces.append((at, n, co, ci))
        at += n + co
    p = used.double().requires_grad_(case["kind"] == "train")

    def conv(l, x):
        at, n, co, ci = pieces[l]
        _, _, stride, up = _layers(case["channels"])[l]
        if up:
            x = F.interpolate(x, scale_factor=2, mode="nearest")
        return F.conv2d(x, p[at:at + n].reshape(co, ci, 3, 3), p[at + n:at + n + co], stride=stride, padding=1)

    x = torch.stack([s["T"], s["R"]], 1).double()
    e0 = torch.relu(conv(0, x))
    e1 = torch.relu(conv(1, e0))
    e2 = torch.relu(conv(2, e1))
    e3 = torch.relu(conv(3, e2))
    d2 = torch.relu(conv(4, e3)) + e2
    d1 = torch.relu(conv(5, d2)) + e1
    v = SCALE * conv(6, d1)
    if case["kind"] == "predict":
        return v
    loss = 0.5 * (v - s["target"].double()).square().mean() / SCALE ** 2
    (g,) = torch.autograd.grad(loss, p)
    return {"grads": g, "params": params.double() - LR * g / (g.abs() + 1e-8)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        return None
    s = _inputs(case, seed)
    if kind in ("predict", "train"):
        return _net64(case, s)
    if kind == "precond":
        return _precond64(case, s["r"])
    T = s["T"]
    tr = _Tracer(case, s["v"], s.get("dv", ()))
    if kind == "forward":
        return _forward64(tr, case, T)
    if kind == "autograd":
        return {"u1": _forward64(tr, case, T), "grad": _jtvp64(tr, case, T, s["r"])}
    if kind == "objective":
        res = _forward64(tr, case, T) - s["R"].double()
        cell = 1.0 / math.prod(tr.im)
        reg = _regularizer(case, s["v"].double())
        D = 0.5 * cell * float(res.square().sum())
        S = 0.5 * float((s["v"].double() * reg).sum())
        return {"J": D + case["alpha"] * S, "D": D, "S": S,
                "grad": _jtvp64(tr, case, T, cell * res) + case["alpha"] * reg}
    out = [h + case["alpha"] * _regularizer(case, dv.double()) + case["gamma"] * dv.double()
           for h, dv in zip(_products64(tr, case, T), s["dv"])]
    return out if kind == "assembled" else out[0]
