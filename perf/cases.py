"""The measured workloads of this framework: effective-field evaluations, time
stepping (RK4, forward Euler, multirate), the adjoint run and the two learned
demag surrogates, each called through the package's public entry points.

Materials are the workload configurations of ``paper_2602_12242_gb300.inputs``
on grids of their own size or of the sizes the tests and the benchmark use.
``exact`` computes the same outputs in FP64 with plain torch (its own Newell
tensor, FFT convolution, stencils, integrators and networks).
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2602_12242_gb300 import autograd, inputs, solver, surrogate

MU0 = 4e-7 * math.pi
D64 = torch.float64


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one effective-field evaluation of a small box: the smallest call (latency, launches)
        dict(name="field_plain", kind="field", base="plain", nx=32, ny=32, nz=4),
        # a monitored run of the small box: ten RK4 steps, then the energies a program logs
        dict(name="rk4_plain_energy", kind="steps", base="plain", nx=32, ny=32, nz=4, method="rk4", steps=10, dt=1e-14,
             energy=True),
        # the thin film with DMI and chiral edges (long runs of an L2-resident grid)
        dict(name="rk4_film", kind="steps", base="film", nx=512, ny=128, nz=1, method="rk4", steps=20, dt=5e-14,
             energy=False),
        # a device-shaped element with odd sizes, three layers, a per-cell Ms map and DMI
        dict(name="rk4_ragged_map", kind="steps", base="adjoint", nx=201, ny=77, nz=3, method="rk4", steps=10,
             dt=1e-14, energy=False),
        # the standard-problem-4 film on its fine grid with the multirate integrator
        dict(name="mri_sp4_fine", kind="steps", base="sp4", nx=640, ny=160, nz=4, method="mri", steps=2, dt=1e-13,
             energy=False),
        # the weak-scaling cube (128^3 cells on one GPU, forward Euler): a deep grid, large transforms along z
        dict(name="euler_cube", kind="steps", base="plain", nx=128, ny=128, nz=128, method="euler", steps=4, dt=1e-15,
             energy=False),
        # the bulk grid with per-grain easy axes: the largest working set, HBM-resident
        dict(name="rk4_bulk", kind="steps", base="bulk", nx=512, ny=512, nz=16, method="rk4", steps=4, dt=1e-14,
             energy=False),
        # gradient of a final-state objective with respect to m0 and the Ms map (forward record and reverse sweep)
        dict(name="adjoint_film", kind="adjoint", base="adjoint", nx=128, ny=128, nz=1, steps=60, every=20, dt=2e-14),
        # the conv-net demag of one field, as an integrator in the loop calls it
        dict(name="conv_field", kind="conv", nx=64, ny=64, nz=4, batch=1, train=False),
        # one training step of the conv net at its training batch
        dict(name="conv_train", kind="conv", nx=64, ny=64, nz=4, batch=64, train=True),
        # the Fourier operator's demag of one film field in the loop
        dict(name="fourier_field", kind="fourier", nx=160, ny=40, modes=12, batch=1, train=False),
        # one training step of the Fourier operator at its training batch
        dict(name="fourier_train", kind="fourier", nx=160, ny=40, modes=12, batch=32, train=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    what = rng.choice(("field", "film", "slab", "cube", "box", "adjoint", "conv", "fourier"))
    if what == "field":
        return dict(kind="field", base=rng.choice(("plain", "bulk", "adjoint")), nx=_log_int(rng, 8, 256),
                    ny=_log_int(rng, 8, 256), nz=_log_int(rng, 1, 16))
    if what == "film":
        return dict(kind="steps", base="film", nx=_log_int(rng, 64, 1000), ny=_log_int(rng, 32, 500), nz=1,
                    method=rng.choice(("rk4", "rk4", "euler")), steps=rng.randint(4, 20), dt=5e-14, energy=False)
    if what == "slab":
        return dict(kind="steps", base=rng.choice(("bulk", "adjoint")), nx=_log_int(rng, 64, 512),
                    ny=_log_int(rng, 64, 512), nz=rng.randint(2, 16), method="rk4", steps=rng.randint(1, 4), dt=1e-14,
                    energy=rng.random() < 0.5)
    if what == "cube":
        n = _log_int(rng, 24, 128)
        return dict(kind="steps", base=rng.choice(("plain", "bulk")), nx=n, ny=max(24, n - rng.randint(0, 9)),
                    nz=max(20, n - rng.randint(0, 30)), method=rng.choice(("rk4", "euler")), steps=rng.randint(1, 4),
                    dt=1e-15, energy=False)
    if what == "box":
        return dict(kind="steps", base="sp4", nx=_log_int(rng, 32, 640), ny=_log_int(rng, 16, 160),
                    nz=rng.randint(1, 6), method="mri", steps=rng.randint(1, 2), dt=5e-14, energy=False)
    if what == "adjoint":
        return dict(kind="adjoint", base="adjoint", nx=rng.randint(24, 128), ny=rng.randint(24, 128),
                    nz=rng.choice((1, 1, 2)), steps=rng.randint(10, 40), every=rng.randint(5, 20), dt=2e-14)
    if what == "conv":
        return dict(kind="conv", nx=rng.randint(20, 64), ny=rng.randint(20, 64), nz=rng.randint(1, 4),
                    batch=_log_int(rng, 1, 64), train=rng.random() < 0.5)
    return dict(kind="fourier", nx=rng.randint(40, 160), ny=rng.randint(36, 64), modes=rng.choice((8, 12, 12, 16)),
                batch=_log_int(rng, 1, 32), train=rng.random() < 0.5)


# the fine standard-problem-4 film (cells of 0.78125 nm); the others are the package's own configurations
_SP4 = dict(dx=0.78125e-9, dy=0.78125e-9, dz=0.78125e-9, Ms=8e5, A=1.3e-11, Ku=0.0, ku_axis=(0.0, 0.0, 1.0), D=0.0,
            dmi=False, alpha=0.02, gamma=2.211e5, h_bias=(-24.6e-3 / MU0, 4.3e-3 / MU0, 0.0))


def _config(case):
    c = dict(_SP4 if case["base"] == "sp4" else inputs.CONFIGS[case["base"]])
    c.update(nx=case["nx"], ny=case["ny"], nz=case["nz"])
    return c


# ---------------------------------------------------------------------------
# Inputs (on the GPU, from the seed alone)
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _record(v):
    """(..., 3) -> contiguous float32 (..., 4) with a zero w slot."""
    return F.pad(v, (0, 1)).float().contiguous()


def _magnetisation(case, seed):
    """Unit vectors (nz, ny, nx, 3): random for the boxes and slabs, near uniform with noise for the films."""
    v = torch.randn(case["nz"], case["ny"], case["nx"], 3, generator=_gen(seed), device="cuda", dtype=D64)
    if case["base"] in ("film", "sp4"):
        d = torch.tensor([1.0, 0.25, 0.1], device="cuda", dtype=D64)
        v = _unit(d) + 0.01 * v
    return _unit(v)


def _maps(case, cfg, seed):
    """(Ms map, easy-axis map) of a case, None where the material has none."""
    shape = (case["nz"], case["ny"], case["nx"])
    ms = axes = None
    if cfg["Ms"] == "map":
        ms = (6e5 + 4e5 * torch.rand(shape, generator=_gen(seed + 1), device="cuda", dtype=D64)).float()
    if cfg["ku_axis"] == "grains":
        gz, gy, gx = 16, 32, 32
        blocks = tuple(-(-n // s) for n, s in zip(shape, (gz, gy, gx)))
        a = _unit(torch.randn(*blocks, 3, generator=_gen(seed + 2), device="cuda", dtype=D64))
        a = a.repeat_interleave(gz, 0).repeat_interleave(gy, 1).repeat_interleave(gx, 2)
        axes = _record(a[:shape[0], :shape[1], :shape[2]])
    return ms, axes


def _context(case, cfg, ms, axes):
    axis = (0.0, 0.0, 1.0) if axes is not None else cfg["ku_axis"]
    ctx = solver.Context(cfg["nx"], cfg["ny"], cfg["nz"], cfg["dx"], cfg["dy"], cfg["dz"],
                         Ms=8e5 if ms is not None else cfg["Ms"], A=cfg["A"], Ku=cfg["Ku"], D=cfg["D"],
                         alpha=cfg["alpha"], gamma=cfg["gamma"], ku_axis=axis, h_bias=cfg["h_bias"], dmi=cfg["dmi"])
    if ms is not None:
        ctx.set_ms_map(ms)
    if axes is not None:
        ctx.set_anis_map(None, axes)
    return ctx


def _textures(shape, sigma, seed):
    """Smooth unit-vector textures (batch, nz, ny, nx, 3): white noise under a periodic Gaussian filter."""
    b, nz, ny, nx = shape
    w = torch.randn(b, 3, nz, ny, nx, generator=_gen(seed), device="cuda", dtype=D64)
    k2 = sum(torch.fft.fftfreq(n, device="cuda", dtype=D64).reshape([-1 if q == a else 1 for q in range(3)]) ** 2
             for a, n in enumerate((nz, ny, nx)))
    f = torch.fft.ifftn(torch.fft.fftn(w, dim=(2, 3, 4)) * torch.exp(-2.0 * (math.pi * sigma) ** 2 * k2),
                        dim=(2, 3, 4)).real
    return _unit(f.movedim(1, -1))


def _pairs(case, seed):
    """(m, demag field) training pairs as float4 records, and the normaliser statistics of the set."""
    if case["kind"] == "conv":
        h, nz = (2e-9, 2e-9, 2e-9), case["nz"]
    else:
        h, nz = (3.125e-9, 3.125e-9, 3.125e-9), 1
    shape = (nz, case["ny"], case["nx"])
    m = _textures((case["batch"],) + shape, 8.0, seed)
    field = _Demag(shape, h)
    t = torch.stack([field(8e5 * x) for x in m])
    stats = []
    for a in (m, t):
        a = a.reshape(-1, 3)
        stats += a.mean(0).tolist() + a.std(0, unbiased=False).tolist()
    return _record(m), _record(t), stats


def _uniform(gen, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=gen, device="cuda", dtype=D64)


def _conv_params(seed):
    gen, parts = _gen(seed + 3), []
    for cin, cout in zip((3, 32, 64, 32), (32, 64, 32, 3)):
        b = 1.0 / math.sqrt(27 * cin)
        parts += [_uniform(gen, cout * cin * 27, -b, b), _uniform(gen, cout, -b, b)]
    return torch.cat(parts).float()


def _fourier_shapes(modes):
    shapes = [(32, 3), (32,)]
    for _ in range(4):
        shapes += [(2 * modes, modes, 32, 32, 2), (32, 32), (32,)]
    return shapes + [(128, 32), (128,), (3, 128), (3,)]


def _fourier_params(modes, seed):
    gen, parts, b = _gen(seed + 3), [], 1.0
    for s in _fourier_shapes(modes):
        n = math.prod(s)
        if len(s) == 5:
            parts.append(_uniform(gen, n, 0.0, 1.0 / 1024))
            continue
        if len(s) == 2:
            b = 1.0 / math.sqrt(s[1])
        parts.append(_uniform(gen, n, -b, b))
    return torch.cat(parts).float()


# ---------------------------------------------------------------------------
# The measured calls
# ---------------------------------------------------------------------------
def prepare(case, seed):
    if case["kind"] in ("conv", "fourier"):
        m, h, stats = _pairs(case, seed)
        if case["kind"] == "conv":
            net = surrogate.Surrogate(case["nx"], case["ny"], case["nz"], case["batch"])
            net.set_params(_conv_params(seed))
        else:
            net = surrogate.FourierSurrogate(case["nx"], case["ny"], case["modes"], case["batch"])
            net.set_params(_fourier_params(case["modes"], seed))
        net.set_normalizer(stats)
        return dict(case=case, net=net, m=m, h=h)
    cfg = _config(case)
    ms, axes = _maps(case, cfg, seed)
    ctx = _context(case, cfg, ms, axes)
    state = dict(case=case, ctx=ctx, m=_record(_magnetisation(case, seed)))
    if case["kind"] == "adjoint":
        ctx.adjoint_reserve(case["steps"], case["every"])
        state["m"].requires_grad_(True)
        state["ms"] = ms.requires_grad_(True)
    return state


def _patch(case):
    """The central quarter of the film, whose mean m_z is the objective."""
    ny, nx = case["ny"], case["nx"]
    return slice(ny * 3 // 8, ny * 5 // 8), slice(nx * 3 // 8, nx * 5 // 8)


def run(state):
    case = state["case"]
    if case["kind"] == "field":
        return state["ctx"].heff(state["m"])
    if case["kind"] == "steps":
        ctx, m = state["ctx"], state["m"]
        ctx.rk_step(m, case["steps"], case["dt"], case["method"])
        return dict(m=m, energy=ctx.energy(m)) if case["energy"] else dict(m=m)
    if case["kind"] == "adjoint":
        m0, ms = state["m"], state["ms"]
        m = autograd.rk4_run(state["ctx"], m0, case["dt"], ms)
        y, x = _patch(case)
        objective = m[:, y, x, 2].mean()
        g_m0, g_ms = torch.autograd.grad(objective, (m0, ms))
        return dict(m=m.detach(), g_m0=g_m0, g_ms=g_ms)
    net = state["net"]
    if not case["train"]:
        return net.forward(state["m"])
    loss, grad = net.loss_grad(state["m"], state["h"])
    net.adam_step(1e-3, 1e-4)
    return dict(loss=loss, grad=grad)


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _pad(n):
    return 1 if n == 1 else 1 << (2 * n - 2).bit_length()


def _demag_work(nx, ny, nz):
    """(flops of one convolution with the zero-padded halves skipped, bytes of the tensor's octant)."""
    px, py, pz = _pad(nx), _pad(ny), _pad(nz)
    hx = px // 2 + 1
    lg = lambda p: math.log2(p) if p > 1 else 0.0  # noqa: E731
    x = 3 * ny * nz * 2.5 * px * lg(px)
    y = 3 * nz * hx * 5.0 * py * lg(py)
    z = 3 * hx * py * 5.0 * pz * lg(pz)
    octant = hx * (py // 2 + 1) * (pz // 2 + 1) * (6 if nz > 1 else 4) * 4
    return 2 * (x + y + z) + 30.0 * hx * py * pz, octant


def work(case):
    nx, ny = case["nx"], case["ny"]
    nz = case.get("nz", 1)
    cells = nx * ny * nz
    if case["kind"] == "conv":
        b, params = case["batch"], 115907
        f = 2.0 * 27 * (3 * 32 + 32 * 64 + 64 * 32 + 32 * 3) * cells * b
        if case["train"]:  # inputs, targets, weights and gradient; forward, data gradient (not of layer 1), weights
            return dict(bytes=32 * cells * b + 28 * params, flops=3 * f - 2.0 * 27 * 96 * cells * b)
        return dict(bytes=32 * cells * b + 4 * params, flops=f)
    if case["kind"] == "fourier":
        b, k = case["batch"], case["modes"]
        params = sum(math.prod(s) for s in _fourier_shapes(k))
        layer = 32 * (4.0 * nx * k * ny + 8.0 * ny * 2 * k * k) * 2 + 8.0 * 32 * 32 * 2 * k * k + 2.0 * 1024 * cells
        f = b * (4 * layer + cells * 2.0 * (3 * 32 + 32 * 128 + 128 * 3))
        return dict(bytes=32 * cells * b + (28 if case["train"] else 4) * params, flops=(3 if case["train"] else 1) * f)
    conv, octant = _demag_work(nx, ny, nz)
    maps = {"bulk": 16, "adjoint": 4}.get(case["base"], 0)
    if case["kind"] == "field":
        return dict(bytes=(32 + maps) * cells + octant, flops=conv + 80.0 * cells)
    if case["kind"] == "adjoint":
        # forward, recomputed stage states and reverse sweep: three convolutions per stage
        n = case["steps"]
        return dict(bytes=(16 * 3 + 8) * cells + octant, flops=n * 4 * (3 * conv + 600.0 * cells))
    evals, local = {"rk4": (4, 4), "euler": (1, 1), "mri": (3, 39)}[case["method"]]
    n = case["steps"]
    return dict(bytes=n * ((32 + maps) * cells + octant), flops=n * (evals * conv + 150.0 * local * cells))


# ---------------------------------------------------------------------------
# FP64 values of the same outputs
# ---------------------------------------------------------------------------
def _newell_f(x, y, z):
    r = torch.sqrt(x * x + y * y + z * z)
    out = (2 * x * x - y * y - z * z) * r / 6
    for a, b in ((y, z), (z, y)):
        d = torch.sqrt(x * x + b * b)
        out = out + torch.where(d > 0, 0.5 * a * (b * b - x * x) * torch.asinh(a / torch.where(d > 0, d, 1.0)), 0.0)
    p = x * r
    return out - torch.where(p != 0, x * y * z * torch.atan(y * z / torch.where(p != 0, p, 1.0)), 0.0)


def _newell_g(x, y, z):
    r = torch.sqrt(x * x + y * y + z * z)
    out = -x * y * r / 3

    def asinh(c, a, d2):
        d = torch.sqrt(d2)
        return torch.where(d > 0, c * torch.asinh(a / torch.where(d > 0, d, 1.0)), 0.0)

    def atan(c, a, p):
        return torch.where(p != 0, c * torch.atan(a / torch.where(p != 0, p, 1.0)), 0.0)

    out = out + asinh(x * y * z, z, x * x + y * y) + asinh(y * (3 * z * z - y * y) / 6, x, y * y + z * z)
    out = out + asinh(x * (3 * z * z - x * x) / 6, y, x * x + z * z) - atan(z ** 3 / 6, x * y, z * r)
    return out - atan(z * y * y / 2, x * z, y * r) - atan(z * x * x / 2, y * z, x * r)


def _second_difference(fn, pos, h):
    """sum of fn over the 27 neighbours of pos, each axis weighted (-1, 2, -1)."""
    out = 0.0
    for i in (-1, 0, 1):
        for j in (-1, 0, 1):
            for k in (-1, 0, 1):
                w = (2.0 if i == 0 else -1.0) * (2.0 if j == 0 else -1.0) * (2.0 if k == 0 else -1.0)
                out = out + w * fn(pos[0] + i * h[0], pos[1] + j * h[1], pos[2] + k * h[2])
    return out


def _tensor_octant(shape, h):
    """The demag tensor (xx, yy, zz, xy, xz, yz) at the non-negative offsets: Newell's closed form near the origin,
    Gauss-Legendre quadrature of its defining integral (a triangle weight per axis) where that form cancels."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    nz, ny, nx = shape
    z, y, x = (torch.arange(n, device=dev, dtype=D64) * s for n, s in zip(shape, (h[2], h[1], h[0])))
    pos = (x[None, None, :], y[None, :, None], z[:, None, None])
    v = h[0] * h[1] * h[2]
    n = torch.zeros((6,) + tuple(shape), device=dev, dtype=D64)
    t, w = np.polynomial.legendre.leggauss(4)
    t, w = 0.5 * (t + 1), 0.5 * w
    nodes = [(s * a, b * (1 - a)) for s in (-1.0, 1.0) for a, b in zip(t, w)]
    for a, wa in nodes:
        for b, wb in nodes:
            for c, wc in nodes:
                q = (pos[0] + a * h[0], pos[1] + b * h[1], pos[2] + c * h[2])
                r2 = q[0] ** 2 + q[1] ** 2 + q[2] ** 2
                s3 = r2.pow_(-1.5).mul_(wa * wb * wc * v / (4 * math.pi))
                s5 = s3 / (q[0] ** 2 + q[1] ** 2 + q[2] ** 2).mul_(-1.0 / 3.0)
                for e, (i, j) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
                    n[e].addcmul_(s5, q[i] * q[j])
                    if i == j:
                        n[e] += s3
    near = 10 * max(h)
    nn = [min(m, int(near / s) + 1) for m, s in zip((nx, ny, nz), h)]
    p = torch.meshgrid(z[:nn[2]], y[:nn[1]], x[:nn[0]], indexing="ij")[::-1]
    inside = p[0] ** 2 + p[1] ** 2 + p[2] ** 2 <= near * near
    order = ((0, 1, 2), (1, 2, 0), (2, 0, 1), (0, 1, 2), (0, 2, 1), (1, 2, 0))
    for e, o in enumerate(order):
        fn = _newell_f if e < 3 else _newell_g
        # lengths in units of the largest cell edge
        u = max(h)
        c = _second_difference(fn, [p[q] / u for q in o], [h[q] / u for q in o]) / (4 * math.pi * v / u ** 3)
        part = n[e, :nn[2], :nn[1], :nn[0]]
        part.copy_(torch.where(inside, c, part))
    return n


class _Demag:
    """H = -N * M by zero-padded FFTs in FP64; M is (nz, ny, nx, 3) in A/m."""

    def __init__(self, shape, h):
        self.shape, self.pad = shape, tuple(_pad(n) for n in shape)
        octant = _tensor_octant(shape, h)
        self.n = []
        for e, odd in enumerate(((), (), (), (1, 2), (0, 2), (0, 1))):  # axes (z, y, x) in which a component is odd
            full = octant[e]
            for axis in range(3):
                m, p = shape[axis], self.pad[axis]
                if m == 1:
                    continue
                gap = list(full.shape)
                gap[axis] = p - (2 * m - 1)
                mirror = full.narrow(axis, 1, m - 1).flip(axis)
                full = torch.cat([full, full.new_zeros(gap), -mirror if axis in odd else mirror], axis)
            self.n.append(torch.fft.rfftn(full).real.contiguous())

    def __call__(self, m):
        nz, ny, nx = self.shape
        s = [torch.fft.rfftn(m[..., c], s=self.pad, dim=(0, 1, 2)) for c in range(3)]
        xx, yy, zz, xy, xz, yz = self.n
        out = []
        for row in ((xx, xy, xz), (xy, yy, yz), (xz, yz, zz)):
            f = sum(a * b for a, b in zip(row, s))
            out.append(-torch.fft.irfftn(f, s=self.pad, dim=(0, 1, 2))[:nz, :ny, :nx])
        return torch.stack(out, -1)


def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


class _Model:
    """Field terms, right-hand side and steps of a case in FP64."""

    def __init__(self, case, cfg, ms, axes):
        self.c, self.ms = cfg, (ms.to(D64)[..., None] if ms is not None else cfg["Ms"])
        self.h = (cfg["dx"], cfg["dy"], cfg["dz"])
        self.demag = _Demag((case["nz"], case["ny"], case["nx"]), self.h)
        e = axes[..., :3].to(D64) if axes is not None else torch.tensor(cfg["ku_axis"], device="cuda", dtype=D64)
        self.axis = e
        self.bias = torch.tensor(cfg["h_bias"], device="cuda", dtype=D64)
        self.kappa = cfg["D"] / (2 * cfg["A"]) if cfg["dmi"] else 0.0

    def _sides(self, m, axis):
        """Fields shifted by +1 and -1 cell along x, y or z, with the ghost cells of the boundary condition."""
        dim = 2 - axis
        first, last = m.narrow(dim, 0, 1), m.narrow(dim, m.shape[dim] - 1, 1)
        if axis < 2:
            k = self.h[axis] * self.kappa
            ez_n = torch.tensor([(0.0, 1.0, 0.0), (-1.0, 0.0, 0.0)][axis], device="cuda", dtype=D64)  # e_z x e_axis
            last, first = last - k * _cross(ez_n.expand_as(last), last), first + k * _cross(ez_n.expand_as(first), first)
        n = m.shape[dim]
        return torch.cat([m.narrow(dim, 1, n - 1), last], dim), torch.cat([first, m.narrow(dim, 0, n - 1)], dim)

    def terms(self, m):
        c, pre = self.c, 1.0 / (MU0 * self.ms)
        sides = [self._sides(m, a) for a in range(3)]
        lap = sum((p + q - 2 * m) / s ** 2 for (p, q), s in zip(sides, self.h))
        t = dict(demag=self.demag(self.ms * m), exch=2 * c["A"] * pre * lap,
                 anis=2 * c["Ku"] * pre * (m * self.axis).sum(-1, keepdim=True) * self.axis, dmi=torch.zeros_like(m),
                 zeeman=self.bias.expand_as(m))
        if c["dmi"]:
            dx, dy = ((sides[a][0] - sides[a][1]) / (2 * self.h[a]) for a in (0, 1))
            t["dmi"] = 2 * c["D"] * pre * torch.stack([dx[..., 2], dy[..., 2], -(dx[..., 0] + dy[..., 1])], -1)
        return t

    def exchange(self, m):
        lap = sum((p + q - 2 * m) / s ** 2 for (p, q), s in ((self._sides(m, a), self.h[a]) for a in range(3)))
        return 2 * self.c["A"] / (MU0 * self.ms) * lap

    def llg(self, m, h):
        mxh = _cross(m, h)
        return -self.c["gamma"] / (1 + self.c["alpha"] ** 2) * (mxh + self.c["alpha"] * _cross(m, mxh))

    def rhs(self, m):
        return self.llg(m, sum(self.terms(m).values()))

    def rk4(self, m, dt):
        k1 = self.rhs(m)
        k2 = self.rhs(_unit(m + 0.5 * dt * k1))
        k3 = self.rhs(_unit(m + 0.5 * dt * k2))
        k4 = self.rhs(_unit(m + dt * k3))
        return m + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4)

    def euler(self, m, dt):
        return m + dt * self.rhs(m)

    def mri(self, m, dt):
        """Explicit-explicit multirate step: Knoth-Wolke on both levels, exchange fast, ten fast steps per unit."""
        a = ((0.0, 0.0, 0.0), (1 / 3, 0.0, 0.0), (-3 / 16, 15 / 16, 0.0), (1 / 6, 3 / 10, 8 / 15))
        c = (0.0, 1 / 3, 3 / 4, 1.0)
        slow, u = [], m
        for i in (1, 2, 3):
            t = self.terms(m)
            slow.append(self.llg(m, t["demag"] + t["anis"] + t["dmi"] + t["zeeman"]))
            dc = c[i] - c[i - 1]
            r = sum((a[i][j] - a[i - 1][j]) / dc * slow[j] for j in range(i))
            n = math.ceil(dc / 0.1 - 1e-9)
            h = dc * dt / n
            for _ in range(n):
                k = []
                for s in range(3):
                    v = _unit(m + h * sum(a[s][j] * k[j] for j in range(s))) if s else m
                    k.append(self.llg(v, self.exchange(v)) + r)
                u = m + h * sum(a[3][j] * k[j] for j in range(3))
                m = _unit(u)
        return u

    def run(self, m, method, steps, dt):
        """The field after `steps` steps, as a record with the norm before the last renormalisation."""
        m = _unit(m)
        u = m
        for _ in range(steps):
            u = getattr(self, method)(m, dt)
            m = _unit(u)
        return torch.cat([m, u.norm(dim=-1, keepdim=True)], -1)

    def energy(self, m):
        c, v = self.c, self.h[0] * self.h[1] * self.h[2]
        t = self.terms(m)
        q = -0.5 * MU0 * v
        e = {k: (q * (self.ms * m * t[k]).sum()).item() for k in ("demag", "exch", "dmi")}
        e["anis"] = (v * c["Ku"] * (1 - (m * self.axis).sum(-1) ** 2)).sum().item()
        e["zeeman"] = (2 * q * (self.ms * m * t["zeeman"]).sum()).item()
        return e


def _gelu(x):
    return 0.5 * x * (1 + torch.erf(x / math.sqrt(2.0)))


def _conv_net(flat, x):
    """x (batch, 3, nz, ny, nx) -> the same shape."""
    o = 0
    for l, (cin, cout) in enumerate(zip((3, 32, 64, 32), (32, 64, 32, 3))):
        w = flat[o:o + cout * cin * 27].reshape(cout, cin, 3, 3, 3)
        o += w.numel()
        b = flat[o:o + cout]
        o += cout
        # one product per tap over channels
        p, y = F.pad(x, (1, 1, 1, 1, 1, 1)), b.reshape(1, -1, 1, 1, 1)
        for k in range(27):
            z, r, s = k // 9, k // 3 % 3, k % 3
            part = p[:, :, z:z + x.shape[2], r:r + x.shape[3], s:s + x.shape[4]]
            y = y + torch.einsum("oi,bizyx->bozyx", w[:, :, z, r, s], part)
        x = _gelu(y) if l < 3 else y
    return x


def _fourier_net(flat, x, modes):
    """x (batch, 3, 1, ny, nx) -> the same shape."""
    x, p, o = x[:, :, 0], [], 0
    for s in _fourier_shapes(modes):
        p.append(flat[o:o + math.prod(s)].reshape(s))
        o += math.prod(s)
    lin = lambda w, b, a: torch.einsum("oi,biyx->boyx", w, a) + b.reshape(1, -1, 1, 1)  # noqa: E731
    v = lin(p[0], p[1], x)
    for l in range(4):
        r, w, b = p[2 + 3 * l:5 + 3 * l]
        s = torch.fft.rfft2(v)
        low, high = s[:, :, :modes, :modes], s[:, :, -modes:, :modes]
        kept = torch.einsum("biyx,yxio->boyx", torch.cat([low, high], 2), torch.view_as_complex(r.contiguous()))
        full = torch.zeros_like(s)
        full[:, :, :modes, :modes] = kept[:, :, :modes]
        full[:, :, -modes:, :modes] = kept[:, :, modes:]
        v = torch.fft.irfft2(full, s=v.shape[-2:]) + lin(w, b, v)
        v = _gelu(v) if l < 3 else v
    return lin(p[-2], p[-1], _gelu(lin(p[-4], p[-3], v)))[:, :, None]


def _exact_net(case, seed):
    m, h, stats = _pairs(case, seed)
    mean, std, hmean, hstd = (torch.tensor(stats[3 * q:3 * q + 3], device="cuda", dtype=D64) for q in range(4))
    conv = case["kind"] == "conv"
    flat = (_conv_params(seed) if conv else _fourier_params(case["modes"], seed)).to(D64)
    x = ((m[..., :3].to(D64) - mean) / std).movedim(-1, 1)
    apply = (lambda a: _conv_net(flat, a)) if conv else (lambda a: _fourier_net(flat, a, case["modes"]))
    if not case["train"]:
        with torch.no_grad():
            y = torch.cat([apply(a) for a in x.split(8)]).movedim(1, -1)
        return F.pad(y * hstd + hmean, (0, 1))
    flat.requires_grad_(True)
    target = ((h[..., :3].to(D64) - hmean) / hstd).movedim(-1, 1)
    loss, grad = 0.0, torch.zeros_like(flat)
    for a, t in zip(x.split(4), target.split(4)):  # a few samples at a time: the saved activations stay small
        part = F.smooth_l1_loss(apply(a), t, reduction="sum") / target.numel()
        loss += part.item()
        grad += torch.autograd.grad(part, flat)[0]
    return dict(loss=torch.tensor([loss], dtype=D64), grad=grad)


def exact(case, seed):
    if case["kind"] in ("conv", "fourier"):
        return _exact_net(case, seed)
    cfg = _config(case)
    ms, axes = _maps(case, cfg, seed)
    if case["kind"] == "adjoint":
        ms = ms.to(D64).requires_grad_(True)
    model = _Model(case, cfg, ms, axes)
    m = _record(_magnetisation(case, seed))[..., :3].to(D64)
    if case["kind"] == "field":
        return F.pad(sum(model.terms(m).values()), (0, 1))
    if case["kind"] == "steps":
        out = model.run(m, case["method"], case["steps"], case["dt"])
        return dict(m=out, energy=model.energy(out[..., :3])) if case["energy"] else dict(m=out)
    m.requires_grad_(True)
    out = model.run(m, "rk4", case["steps"], case["dt"])
    y, x = _patch(case)
    g_m0, g_ms = torch.autograd.grad(out[:, y, x, 2].mean(), (m, ms))
    return dict(m=out.detach(), g_m0=F.pad(g_m0, (0, 1)), g_ms=g_ms)
