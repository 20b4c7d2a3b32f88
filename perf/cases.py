"""The work that users of this framework have it do, as cases to be timed.

Each case is one pass through the public binding (paper_1406_7459_gb300.mm)
on state that a program would hold: a solver context, a batch or a network,
and a magnetisation.  `listed()` gives the cases themselves, `draw()` more of
the same ranges, `prepare()` the state, `run()` one pass, `work()` what the
pass cannot do without, and `exact()` the same results in 64 bits by plain
torch (an independent demag tensor, FFT convolution, integrators and FNO).

Kinds
  film, block   a block of steps between two outputs of a simulation: set the
                state, n steps (Euler, Heun or RK4), read the state, and with
                "energy" the energies that a relaxation is followed by
  adaptive      an error-controlled run over a span of time
  host          the state lives in page-locked host memory: the whole call
  batch         many uneven samples stepped together
  fno           the surrogate's forward pass, or its loss and gradients
"""
import math
import random

import numpy as np
import torch

from paper_1406_7459_gb300 import inputs, mm

MS, A_EX, GAMMA = 8.6e5, 1.3e-11, inputs.GAMMA0
MU0 = 4e-7 * math.pi

# cell (m), Ku, alpha, H_ext and dt of the workloads of inputs.py: the thin
# film (relaxing from a random state), the size sweep and reversal film, and
# the relaxing cube
MATERIALS = {
    "thin": dict(cell=(5e-9, 5e-9, 3e-9), Ku=0.0, alpha=0.5, H=(0.0, 0.0, 0.0), dt=1e-13, start="random"),
    "sweep": dict(cell=(4e-9, 4e-9, 4e-9), Ku=5e2, alpha=0.02, H=inputs.field_at_angle(2.5e4, 170.0), dt=5e-14,
                  start="perturbed"),
    "cube": dict(cell=(4e-9, 4e-9, 4e-9), Ku=5e2, alpha=0.5, H=(0.0, 0.0, 0.0), dt=5e-14, start="random"),
}


def _grid_case(kind, grid, material, **more):
    return dict(kind=kind, nx=grid[0], ny=grid[1], nz=grid[2], material=material, **more)


def listed():
    def case(name, *a, **k):
        return dict(_grid_case(*a, **k), name=name)

    return [
        # the smallest film of the configurations: launches and latency count
        case("film-32x32x1", "film", (32, 32, 1), "thin", method="euler", steps=100, energy=False),
        # the benchmark film, the state kept on the device between blocks of steps
        case("film-256x256x4", "film", (256, 256, 4), "sweep", method="euler", steps=20, energy=False),
        # the largest film of the size sweep
        case("film-512x512x8", "film", (512, 512, 8), "sweep", method="euler", steps=4, energy=False),
        # the sweep's film whose sides are no powers of two, relaxed and its energies read
        case("film-200x60x3", "film", (200, 60, 3), "sweep", method="euler", steps=20, energy=True),
        # a wide single layer with ragged sides under the fourth-order stepper
        case("film-600x400x1-rk4", "film", (600, 400, 1), "thin", method="rk4", steps=4, energy=False),
        # a thick sample whose sides are no powers of two
        case("block-100x80x20", "block", (100, 80, 20), "cube", method="euler", steps=10, energy=True),
        # the largest cube of the paper's Table 1 curve
        case("cube-128", "block", (128, 128, 128), "cube", method="euler", steps=4, energy=False),
        # an error-controlled run
        case("adaptive-128x128x4", "adaptive", (128, 128, 4), "sweep", span=1e-12, tol=1e-4),
        # the benchmark film stepped from and to host memory
        case("host-256x256x4", "host", (256, 256, 4), "sweep", steps=1),
        # the 512 uneven samples of the batch workload
        dict(name="batch-512", kind="batch", samples=512, mix=3, steps=10),
        # the surrogate of the benchmark: one increment forward; a training batch's gradients
        dict(name="fno-forward-256", kind="fno", H=256, W=256, width=32, modes=16, layers=4, batch=1, grad=False),
        dict(name="fno-grad-256", kind="fno", H=256, W=256, width=32, modes=16, layers=4, batch=8, grad=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi):
    """A side of lo..hi cells: mostly any size, now and then a power of two."""
    n = _log_int(rng, lo, hi)
    return 1 << round(math.log2(n)) if rng.random() < 0.25 else n


_EVALS = {"euler": 1, "heun": 2, "rk4": 4}


def draw(rng):
    kind = rng.choice(["film", "film", "film", "block", "block", "adaptive", "host", "batch", "fno", "fno"])
    if kind == "film":
        while True:
            g = (_side(rng, 16, 1024), _side(rng, 16, 1024), rng.choice((1, 1, 2, 3, 4, 5, 8)))
            if g[0] * g[1] * g[2] <= 1 << 20:
                break
        method = rng.choice(("euler", "euler", "heun", "rk4"))
        steps = max(1, min(60, (1 << 21) // (g[0] * g[1] * g[2] * _EVALS[method])))
        return _grid_case(kind, g, rng.choice(("thin", "sweep")), method=method, steps=steps,
                          energy=rng.random() < 0.3)
    if kind == "block":
        while True:
            g = (_side(rng, 8, 160), _side(rng, 8, 160), _side(rng, 10, 128))
            if g[0] * g[1] * g[2] <= 1 << 20:
                break
        steps = max(1, min(20, (1 << 20) // (g[0] * g[1] * g[2])))
        return _grid_case(kind, g, "cube", method=rng.choice(("euler", "euler", "rk4")) if steps > 4 else "euler",
                          steps=max(1, steps // 4), energy=rng.random() < 0.3)
    if kind == "adaptive":
        while True:
            g = (_side(rng, 16, 256), _side(rng, 16, 256), rng.choice((1, 2, 3, 4)))
            if g[0] * g[1] * g[2] <= 1 << 16:
                break
        return _grid_case(kind, g, "sweep", span=rng.choice((5e-13, 1e-12)), tol=1e-4)
    if kind == "host":
        while True:
            g = (_side(rng, 32, 512), _side(rng, 32, 512), rng.choice((1, 2, 3, 4)))
            if g[0] * g[1] * g[2] <= 1 << 18:
                break
        return _grid_case(kind, g, "sweep", steps=rng.choice((1, 1, 4)))
    if kind == "batch":
        return dict(kind=kind, samples=_log_int(rng, 8, 400), mix=rng.randrange(10, 1 << 20), steps=rng.randint(2, 10))
    modes = rng.choice((4, 8, 12, 16))
    grad = rng.random() < 0.5
    return dict(kind="fno", H=_log_int(rng, max(32, 2 * modes), 256), W=_log_int(rng, max(48, 2 * modes + 1), 256),
                width=rng.choice((8, 16, 32)), modes=modes, layers=rng.choice((2, 4)),
                batch=rng.randint(1, 8) if grad else rng.choice((1, 1, 2, 4)), grad=grad)


# ------------------------------------------------------------- inputs --
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _start(grid, start, gen):
    """|M| = Ms: random directions, or +x with a perturbation of 0.1 per
    component; FP32, (3, nz, ny, nx)."""
    nx, ny, nz = grid
    v = torch.randn((3, nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64)
    if start == "perturbed":
        v *= 0.1
        v[0] += 1.0
    v *= MS / v.square().sum(0).sqrt()
    return v.float()


def _case_start(case, seed):
    m = MATERIALS[case["material"]]
    return _start((case["nx"], case["ny"], case["nz"]), m["start"], _generator(seed))


def _batch_samples(case):
    """Uneven samples as the batch workload has them: 16..256 x 16..64 x 1..2
    cells, each with its own anisotropy, damping and field."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["samples"]):
        d = [rng.gauss(0, 1) for _ in range(3)]
        h = rng.uniform(0, 5e4) / math.sqrt(sum(x * x for x in d))
        out.append(dict(grid=(rng.randint(16, 256), rng.randint(16, 64), rng.randint(1, 2)), Ku=rng.uniform(0, 1e4),
                        alpha=rng.uniform(0.01, 0.5), H=tuple(h * x for x in d)))
    return out


BATCH_CELL, BATCH_DT = (5e-9, 5e-9, 3e-9), 5e-14


def _batch_start(case, seed):
    gen = _generator(seed)
    return [_start(s["grid"], "random", gen) for s in _batch_samples(case)]


def _fno_inputs(case, seed):
    """Weights at the network's own initial scale with small biases, unit-scale
    increments x and targets t of the same scale."""
    gen = _generator(seed)
    C, m, L, B, H, W = (case[k] for k in ("width", "modes", "layers", "batch", "H", "W"))

    def normal(shape, scale):
        return scale * torch.randn(shape, generator=gen, device="cuda")

    p = {"P": normal((C, 5), 5 ** -0.5), "p": normal((C,), 0.05), "R_re": normal((L, C, C, 2 * m, m), 1 / C),
         "R_im": normal((L, C, C, 2 * m, m), 1 / C), "W": normal((L, C, C), C ** -0.5), "b": normal((L, C), 0.05),
         "Q": normal((3, C), C ** -0.5), "q": normal((3,), 0.05)}
    return p, normal((B, 3, H, W), 1.0), normal((B, 3, H, W), 1.0)


# ------------------------------------------------------ prepare and run --
class State:
    pass


def prepare(case, seed):
    s = State()
    s.case = case
    if case["kind"] == "fno":
        p, s.x, s.t = _fno_inputs(case, seed)
        s.net = mm.mm_fno_create(case["H"], case["W"], case["width"], case["modes"], case["layers"],
                                 max_batch=case["batch"])
        flat = torch.cat([v.reshape(-1) for v in p.values()])
        mm.mm_fno_set_params(s.net, flat)
        s.out = torch.empty_like(flat) if case["grad"] else torch.empty_like(s.x)
        return s
    if case["kind"] == "batch":
        samples = _batch_samples(case)
        n = len(samples)
        s.batch = mm.mm_batch_create([x["grid"] for x in samples], [BATCH_CELL] * n, [MS] * n, [A_EX] * n,
                                     [x["Ku"] for x in samples], [x["alpha"] for x in samples], [GAMMA] * n)
        mm.mm_batch_set_field(s.batch, [x["H"] for x in samples])
        s.M = torch.cat([v.reshape(-1) for v in _batch_start(case, seed)])
        s.out = torch.empty_like(s.M)
        return s
    m = MATERIALS[case["material"]]
    s.ctx = mm.mm_create((case["nx"], case["ny"], case["nz"]), m["cell"], MS, A_EX, m["Ku"], m["alpha"], GAMMA)
    mm.mm_set_field(s.ctx, m["H"])
    if case.get("method", "euler") != "euler":
        mm.mm_set_integrator(s.ctx, case["method"])
    s.dt = m["dt"]
    s.M = _case_start(case, seed).reshape(-1)
    s.out = torch.empty_like(s.M)
    if case["kind"] == "host":
        s.M, s.out = s.M.cpu().pin_memory(), s.out.cpu().pin_memory()
    return s


def run(s):
    case = s.case
    if case["kind"] == "fno":
        if case["grad"]:
            loss = mm.mm_fno_grad(s.net, s.x, s.t, s.out)
            return {"loss": loss, "grad": s.out}
        return mm.mm_fno_forward(s.net, s.x, s.out)
    if case["kind"] == "batch":
        mm.mm_batch_set_m(s.batch, s.M)
        mm.mm_batch_step(s.batch, case["steps"], BATCH_DT)
        return mm.mm_batch_get_m(s.batch, s.out)
    if case["kind"] == "host":
        return mm.mm_step_host(s.ctx, s.M, case["steps"], s.dt, s.out)
    mm.mm_set_m(s.ctx, s.M)
    if case["kind"] == "adaptive":
        _, _, stats = mm.mm_run_adaptive(s.ctx, case["span"], s.dt, case["tol"])
        return {"M": mm.mm_get_m(s.ctx, s.out), "accepted": stats["accepted"], "rejected": stats["rejected"]}
    mm.mm_step(s.ctx, case["steps"], s.dt)
    out = {"M": mm.mm_get_m(s.ctx, s.out)}
    if case["energy"]:
        # sums of an FP32 state and its FP32 field: plain numbers, not 64-bit results
        out["E"] = [float(e) for e in mm.mm_energy(s.ctx)]
    return out


# ----------------------------------------------------------------- work --
def _field_work(grid):
    """One field evaluation and update of an n-cell sample: the state in and
    out, the real octant of the tensor spectrum; FFT flops of the padded
    half-spectra there and back (5 L log2 L per transform, half of it for real
    data and for the zero half) and ~60 per cell for the product and update."""
    n = grid[0] * grid[1] * grid[2]
    octant = math.prod((g if g > 1 else 0) + 1 for g in grid)
    padded = math.prod(2 * g if g > 1 else 1 for g in grid)
    logs = sum(math.log2(2 * g) for g in grid if g > 1)
    return 24 * n + 24 * octant, 6 * 2.5 * padded * logs / 2 + 60 * n


def work(case):
    if case["kind"] == "fno":
        C, m, L, B, H, W = (case[k] for k in ("width", "modes", "layers", "batch", "H", "W"))
        px = B * H * W
        params = 9 * C + 3 + L * (C * C * 4 * m * m + C * C + C)
        per_layer = px * 2 * C * C + 2 * (B * C * (H * 2 * W * 2 * m + 8 * H * 2 * m * m)) + B * C * C * 2 * m * m * 8
        flops = L * per_layer + px * 16 * C
        if case["grad"]:
            return {"bytes": 4 * (2 * params + 6 * px), "flops": 3 * flops}
        return {"bytes": 4 * (params + 6 * px), "flops": flops}
    if case["kind"] == "batch":
        each = [_field_work(s["grid"]) for s in _batch_samples(case)]
        return {"bytes": case["steps"] * sum(b for b, _ in each), "flops": case["steps"] * sum(f for _, f in each)}
    b, f = _field_work((case["nx"], case["ny"], case["nz"]))
    if case["kind"] == "adaptive":
        evals = 13                      # at least two trial steps: 1 + 6 each
    else:
        evals = case["steps"] * _EVALS[case.get("method", "euler")] + (1 if case.get("energy") else 0)
    return {"bytes": evals * b, "flops": evals * f}


# ---------------------------------------------------------------- exact --
# Everything below is float64 torch and numpy only.
def _newell_f(x, y, z):
    x2, y2, z2 = x * x, y * y, z * z
    R = (x2 + y2 + z2).sqrt()

    def ratio(a, b):
        return torch.where(b != 0, a / torch.where(b != 0, b, torch.ones_like(b)), torch.zeros_like(b))

    return ((2 * x2 - y2 - z2) * R / 6 + 0.5 * y * (z2 - x2) * torch.asinh(ratio(y, (x2 + z2).sqrt()))
            + 0.5 * z * (y2 - x2) * torch.asinh(ratio(z, (x2 + y2).sqrt())) - x * y * z * torch.atan(ratio(y * z, x * R)))


def _newell_g(x, y, z):
    x2, y2, z2 = x * x, y * y, z * z
    R = (x2 + y2 + z2).sqrt()

    def ratio(a, b):
        return torch.where(b != 0, a / torch.where(b != 0, b, torch.ones_like(b)), torch.zeros_like(b))

    return (-x * y * R / 3 + x * y * z * torch.asinh(ratio(z, (x2 + y2).sqrt()))
            + y / 6 * (3 * z2 - y2) * torch.asinh(ratio(x, (y2 + z2).sqrt()))
            + x / 6 * (3 * z2 - x2) * torch.asinh(ratio(y, (x2 + z2).sqrt()))
            - z * z2 / 6 * torch.atan(ratio(x * y, z * R)) - z * y2 / 2 * torch.atan(ratio(x * z, y * R))
            - z * x2 / 2 * torch.atan(ratio(y * z, x * R)))


def _near(X, Y, Z, cell):
    """Newell's closed form of the cell-to-cell tensor (xx, xy, xz, yy, yz, zz)."""
    out = [0.0] * 6
    for ex in (-1, 0, 1):
        for ey in (-1, 0, 1):
            for ez in (-1, 0, 1):
                w = (2 if ex == 0 else -1) * (2 if ey == 0 else -1) * (2 if ez == 0 else -1)
                a, b, c = X + ex * cell[0], Y + ey * cell[1], Z + ez * cell[2]
                for i, v in enumerate((_newell_f(a, b, c), _newell_g(a, b, c), _newell_g(a, c, b), _newell_f(b, a, c),
                                       _newell_g(b, c, a), _newell_f(c, b, a))):
                    out[i] = out[i] + w * v
    return torch.stack(out) / (4 * math.pi * math.prod(cell))


def _far(X, Y, Z, cell, nodes):
    """The same average by Gauss-Legendre quadrature of the dipole tensor."""
    t, w = np.polynomial.legendre.leggauss(nodes)
    t, w = 0.5 * (t + 1), 0.5 * w
    rule = [(sign * s, q * (1 - s)) for sign in (1, -1) for s, q in zip(t, w)]
    out = torch.zeros((6,) + X.shape, dtype=torch.float64, device=X.device)
    for ax, wx in rule:
        for ay, wy in rule:
            for az, wz in rule:
                a, b, c = X + ax * cell[0], Y + ay * cell[1], Z + az * cell[2]
                r2 = a * a + b * b + c * c
                q = wx * wy * wz / (r2 * r2 * r2.sqrt())
                for i, v in enumerate((r2 - 3 * a * a, -3 * a * b, -3 * a * c, r2 - 3 * b * b, -3 * b * c,
                                       r2 - 3 * c * c)):
                    out[i] += v * q
    return out * (math.prod(cell) / (4 * math.pi))


def _octant(grid, cell):
    """The demag tensor at offsets (i, j, k) >= 0: (6, nz, ny, nx)."""
    k, j, i = torch.meshgrid(*(torch.arange(n, dtype=torch.float64, device="cuda") for n in reversed(grid)),
                             indexing="ij")
    X, Y, Z = (v.reshape(-1) * d for v, d in zip((i, j, k), cell))
    far = (X * X + Y * Y + Z * Z).sqrt() / max(cell)
    out = torch.empty((6, X.numel()), dtype=torch.float64, device="cuda")
    for lo, hi, nodes in ((-1, 8, 0), (8, 16, 5), (16, 32, 4), (32, math.inf, 3)):
        at = ((far >= lo) & (far < hi)).nonzero()[:, 0]
        if at.numel():
            p = X[at], Y[at], Z[at]
            out[:, at] = _far(*p, cell, nodes) if nodes else _near(*p, cell)
    return out.reshape((6,) + tuple(reversed(grid)))


# sign of each component when x, y or z of the offset changes sign
_ODD = ((), (0, 1), (0, 2), (), (1, 2), ())


class _Sample:
    """One sample's field and integrators in 64 bits."""

    def __init__(self, grid, cell, Ku, alpha, H, octant=None):
        self.grid, self.cell, self.Ku, self.alpha = grid, cell, Ku, alpha
        self.H = torch.tensor(H, dtype=torch.float64, device="cuda").reshape(3, 1, 1, 1)
        N = _octant(grid, cell) if octant is None else octant
        self.L = tuple(2 * n if n > 1 else 1 for n in reversed(grid))          # z, y, x
        spectra = []
        for c in range(6):
            t = -N[c]
            for axis, n in ((0, grid[2]), (1, grid[1]), (2, grid[0])):
                if n > 1:
                    odd = (2 - axis) in _ODD[c]
                    back = t.narrow(axis, 1, n - 1).flip(axis) * (-1.0 if odd else 1.0)
                    t = torch.cat([t, torch.zeros_like(t.narrow(axis, 0, 1)), back], axis)
            spectra.append(torch.fft.rfftn(t).real.contiguous())
        self.K = spectra

    def demag(self, M):
        nx, ny, nz = self.grid
        F = [torch.fft.rfftn(M[c], s=self.L) for c in range(3)]
        K = self.K
        rows = ((0, 1, 2), (1, 3, 4), (2, 4, 5))
        return torch.stack([torch.fft.irfftn(sum(K[r[b]] * F[b] for b in range(3)), s=self.L)[:nz, :ny, :nx]
                            for r in rows])

    def field(self, M):
        H = self.demag(M) + self.H
        pref = 2 * A_EX / (MU0 * MS * MS)
        for axis, d in ((3, self.cell[0]), (2, self.cell[1]), (1, self.cell[2])):
            n = M.shape[axis]
            if n > 1:
                step = (M.narrow(axis, 1, n - 1) - M.narrow(axis, 0, n - 1)) * (pref / d ** 2)
                H.narrow(axis, 0, n - 1).add_(step)
                H.narrow(axis, 1, n - 1).sub_(step)
        H[1:] += (-2 * self.Ku / (MU0 * MS * MS)) * M[1:]
        return H

    def rhs(self, M):
        MxH = torch.linalg.cross(M, self.field(M), dim=0)
        c = GAMMA / (1 + self.alpha ** 2)
        return -c * MxH - (c * self.alpha / MS) * torch.linalg.cross(M, MxH, dim=0)

    @staticmethod
    def unit(M):
        return M * (MS / M.square().sum(0).sqrt())

    def step(self, M, dt, method="euler"):
        f = self.rhs
        k1 = f(M)
        if method == "euler":
            return self.unit(M + dt * k1)
        if method == "heun":
            return self.unit(M + 0.5 * dt * (k1 + f(M + dt * k1)))
        k2 = f(M + 0.5 * dt * k1)
        k3 = f(M + 0.5 * dt * k2)
        return self.unit(M + dt / 6 * (k1 + 2 * k2 + 2 * k3 + f(M + dt * k3)))

    def adaptive(self, M, span, dt, tol):
        """Dormand-Prince RK5(4), J. Comput. Appl. Math. 6 (1980) 19-26, with
        the step control that mm_run_adaptive documents."""
        a = ((1 / 5,), (3 / 40, 9 / 40), (44 / 45, -56 / 15, 32 / 9),
             (19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729),
             (9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656),
             (35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84))
        e = (71 / 57600, 0, -71 / 16695, 71 / 1920, -17253 / 339200, 22 / 525, -1 / 40)
        t, accepted, rejected, after = 0.0, 0, 0, False
        k1 = self.rhs(M)
        while span - t > 1e-12 * span:
            h, k = min(dt, span - t), [k1]
            for i, row in enumerate(a):
                Y = M + h * sum(w * q for w, q in zip(row, k) if w)
                Y = self.unit(Y) if i == 5 else Y
                k.append(self.rhs(Y))
            err = float((h * sum(w * q for w, q in zip(e, k) if w)).square().sum(0).sqrt().max()) / MS
            factor = min(5.0, max(0.2, 0.9 * (tol / err) ** 0.2 if err > 0 else 5.0))
            if err <= tol:
                t, M, k1, accepted = t + h, Y, k[6], accepted + 1
                dt, after = h * (min(factor, 1.0) if after else factor), False
            else:
                rejected += 1
                dt, after = h * min(factor, 1.0), True
        return M, accepted, rejected

    def energies(self, M):
        V, m = math.prod(self.cell), M / MS
        ex = sum(float((m.narrow(x, 1, m.shape[x] - 1) - m.narrow(x, 0, m.shape[x] - 1)).square().sum()) / d ** 2
                 for x, d in ((3, self.cell[0]), (2, self.cell[1]), (1, self.cell[2])))
        E = [A_EX * V * ex, self.Ku * V * float(m[1:].square().sum()), -0.5 * MU0 * V * float((self.demag(M) * M).sum()),
             -MU0 * V * float((self.H * M).sum())]
        return [sum(E)] + E


def _fno_forward(p, x, modes):
    B, _, H, W = x.shape
    ky = torch.cat([torch.arange(modes), torch.arange(H - modes, H)]).cuda()
    yy = (torch.arange(H, dtype=torch.float64, device="cuda") / H).reshape(1, 1, H, 1).expand(B, 1, H, W)
    xx = (torch.arange(W, dtype=torch.float64, device="cuda") / W).reshape(1, 1, 1, W).expand(B, 1, H, W)
    v = torch.einsum("oc,bchw->bohw", p["P"], torch.cat([x, yy, xx], 1)) + p["p"].reshape(-1, 1, 1)
    L = p["W"].shape[0]
    for layer in range(L):
        vh = torch.fft.rfft2(v)[:, :, ky, :modes]
        w = torch.einsum("coyx,bcyx->boyx", torch.complex(p["R_re"][layer], p["R_im"][layer]), vh)
        full = torch.zeros(v.shape[:2] + (H, W // 2 + 1), dtype=torch.complex128, device="cuda")
        full[:, :, ky, :modes] = w
        v = torch.fft.irfft2(full, s=(H, W)) + torch.einsum("oc,bchw->bohw", p["W"][layer], v) + p["b"][layer].reshape(
            -1, 1, 1)
        if layer < L - 1:
            v = torch.nn.functional.gelu(v)
    return torch.einsum("oc,bchw->bohw", p["Q"], v) + p["q"].reshape(-1, 1, 1)


def exact(case, seed):
    if case["kind"] == "fno":
        p, x, t = _fno_inputs(case, seed)
        p = {k: v.double().requires_grad_(case["grad"]) for k, v in p.items()}
        y = _fno_forward(p, x.double(), case["modes"])
        if not case["grad"]:
            return y
        loss = (y - t.double()).square().mean()
        grads = torch.autograd.grad(loss, list(p.values()))
        return {"loss": float(loss), "grad": torch.cat([g.reshape(-1) for g in grads])}
    if case["kind"] == "batch":
        samples, out = _batch_samples(case), []
        N = _octant(tuple(max(s["grid"][a] for s in samples) for a in range(3)), BATCH_CELL)
        for s, M in zip(samples, _batch_start(case, seed)):
            nx, ny, nz = s["grid"]
            one, M = _Sample(s["grid"], BATCH_CELL, s["Ku"], s["alpha"], s["H"], N[:, :nz, :ny, :nx]), M.double()
            for _ in range(case["steps"]):
                M = one.step(M, BATCH_DT)
            out.append(M.reshape(-1))
        return torch.cat(out)
    m = MATERIALS[case["material"]]
    one = _Sample((case["nx"], case["ny"], case["nz"]), m["cell"], m["Ku"], m["alpha"], m["H"])
    M = _case_start(case, seed).double()
    if case["kind"] == "adaptive":
        M, accepted, rejected = one.adaptive(M, case["span"], m["dt"], case["tol"])
        return {"M": M.reshape(-1), "accepted": accepted, "rejected": rejected}
    for _ in range(case["steps"]):
        M = one.step(M, m["dt"], case.get("method", "euler"))
    if case["kind"] == "host":
        return M.reshape(-1)
    out = {"M": M.reshape(-1)}
    if case["energy"]:
        out["E"] = one.energies(M)
    return out
