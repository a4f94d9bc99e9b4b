"""The work that users have this library do, as cases that can be timed and compared.

A case is a dict of plain values.  ``kind`` names the call; the other keys are its sizes:

  sample   twa_sample: the Wigner ensemble of a coherent state
  run      twa_run: sample, then step with moments every few steps (a whole call)
  advance  twa_advance of a batch in hand: steps with moments every few steps
  step     twa_step_batch of a batch in hand
  dataset  twa_step_batch, then twa_moments of every instance (what makes training data)
  moments  twa_moments with every output
  phases   twa_phase_moments with every output
  forward  the surrogate's forward pass
  train    one training step of the surrogate (forward, loss, backward, AdamW)

Grids are texts ("128x128x128", several instances joined by "+"), stream counts are texts joined the
same way.  Fields and weights come from torch generators seeded with the case's seed, on the GPU.
``exact`` is the same mathematics in 64 bits with torch alone.
"""
import math

import torch

from paper_2310_07119_gb300 import Ensemble, F32, F64_PLAIN, twa_phase_moments, twa_sample
from paper_2310_07119_gb300 import twa_run
from paper_2310_07119_gb300.fno import FNO

COUPLING = 4.0 * math.pi     # lap V = C |psi|^2 with the dynamical time 1
HBAR = 0.0122                # hbar / m of the 2D and 3D systems (the 1D system has 1)
SCALARS = 8


# --------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # drawing the ensemble of a 3D run: every run begins with it
        {"name": "sample_3d", "kind": "sample", "grids": "128x128x128", "streams": "64", "n_tot": 1e9},
        # the 1D test problem from its classical field to its scalar series, one call
        {"name": "run_1d", "kind": "run", "grids": "256", "streams": "32", "steps": 1000, "every": 10, "n_tot": 1e4},
        # the same system on the plain FP64 path, which checks the FP32 one
        {"name": "advance_1d_f64", "kind": "advance", "grids": "256", "streams": "32", "steps": 100, "every": 10,
         "n_tot": 1e4, "f64": True},
        # the 2D merger at three resolutions in one handle
        {"name": "advance_2d_mix", "kind": "advance", "grids": "512x512+1024x1024+2048x2048", "streams": "128+64+16",
         "steps": 20, "every": 10, "n_tot": 1e9},
        # the 3D condensation ensemble with moments every 10 steps (the benchmark's workload)
        {"name": "advance_3d", "kind": "advance", "grids": "128x128x128", "streams": "256", "steps": 20, "every": 10,
         "n_tot": 1e9},
        # the 3D stable object: larger lines, no moments on the way
        {"name": "step_3d_256", "kind": "step", "grids": "256x256x256", "streams": "64", "steps": 5, "n_tot": 1e10},
        # one snapshot of the surrogate's training data: small grids, many short launches
        {"name": "dataset_3d_32", "kind": "dataset", "grids": "32x32x32+32x32x32", "streams": "8+64", "steps": 50,
         "n_tot": 1e9},
        # one stream of the 3D system on the plain FP64 path
        {"name": "step_3d_f64", "kind": "step", "grids": "128x128x128", "streams": "1", "steps": 2, "n_tot": 1e9,
         "f64": True},
        # every moment of a finished 3D run
        {"name": "moments_3d", "kind": "moments", "grids": "128x128x128", "streams": "256", "n_tot": 1e9},
        # amplitude and phase variances of a finished 3D run
        {"name": "phases_3d", "kind": "phases", "grids": "128x128x128", "streams": "64", "n_tot": 1e9},
        # predicting two correction spectra of the 128^3 system
        {"name": "fno_forward", "kind": "forward", "grid": 128, "width": 32, "modes": 16, "layers": 4, "batch": 2},
        # one training step at 64^3
        {"name": "fno_train", "kind": "train", "grid": 64, "width": 32, "modes": 16, "layers": 4, "batch": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _axes(rng, dim, most):
    """Powers of two from 8, at most `most` cells together and 2048 cells an axis (256 in 3D)."""
    while True:
        a = [2 ** rng.randint(3, {1: 11, 2: 11, 3: 8}[dim]) for _ in range(dim)]
        if math.prod(a) <= most:
            return a


def _text(axes):
    return "x".join(str(v) for v in axes)


def draw(rng):
    kind = rng.choice(["sample", "run", "advance", "advance", "advance", "step", "step", "dataset", "moments", "phases",
                       "forward", "train"])
    if kind in ("forward", "train"):
        while True:
            grid, modes = _log_int(rng, 8, 128), rng.randint(1, 16)
            width, layers, batch = rng.choice([8, 16, 20, 32, 32, 48, 64]), rng.randint(1, 4), _log_int(rng, 1, 8)
            weights = layers * (2 * modes) ** 3 * width ** 2 * 2
            if 2 * (2 * modes) ** 3 <= grid ** 3 and weights <= 3e8 and batch * width * layers * grid ** 3 <= 2.7e8:
                return {"kind": kind, "grid": grid, "width": width, "modes": modes, "layers": layers, "batch": batch}
    f64 = kind in ("advance", "step") and rng.random() < 0.3
    n = rng.randint(1, 3) if kind == "advance" and not f64 and rng.random() < 0.4 else 2 if kind == "dataset" else 1
    dim = rng.randint(1, 3)
    if kind == "dataset":
        axes = [[2 ** rng.randint(4, 6)] * 3] * n
    elif kind == "run":
        axes = [_axes(rng, 1, 2048)]
    else:
        axes = [_axes(rng, dim, 2 ** 21 if f64 else 2 ** 24) for _ in range(n)]
    values = 3e7 if f64 else 2.7e8 / n     # field values of one instance at most
    streams = [_log_int(rng, 1, max(1, min(16 if f64 else 256, values / math.prod(a) - 1))) for a in axes]
    case = {"kind": kind, "grids": "+".join(_text(a) for a in axes), "streams": "+".join(str(s) for s in streams),
            "n_tot": 10.0 ** rng.uniform(8, 10) if len(axes[0]) > 1 else 10.0 ** rng.uniform(4, 8)}
    if kind in ("run", "advance", "step", "dataset"):
        total = sum((s + 1) * math.prod(a) for s, a in zip(streams, axes))
        most = min(400 // (streams[0] + 1) + 4 if f64 else 500, max(4, 4e9 / total))
        case["steps"] = _log_int(rng, 1, most)
    if kind in ("run", "advance"):
        case["every"] = rng.choice([1, 2, 5, 10])
        case["steps"] = max(1, case["steps"] // case["every"]) * case["every"]
    if f64:
        case["f64"] = True
    return case


# ------------------------------------------------------------------------------- sizes and physics
def _instances(case):
    """[(nx, ny, nz)[:dim], streams] of every instance."""
    return [([int(v) for v in g.split("x")], int(s))
            for g, s in zip(case["grids"].split("+"), case["streams"].split("+"))]


def _physics(case):
    """hbar / m, the time step: pi / 4 of kinetic phase at most, as the workloads have it."""
    axes = [a for a, _ in _instances(case)]
    if len(axes[0]) == 1:
        return 1.0, 1e-3
    # 2D instances of several sizes share the step of a 2048 x 2048 grid
    k2 = max(sum((math.pi * n) ** 2 for n in ([2048, 2048] if len(a) == 2 else a)) for a in axes)
    return HBAR, (math.pi / 4.0) * 2.0 / (HBAR * k2)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _k2(axes):
    """|k|^2 on the FFT grid, shape (.., ny, nx), box side 1."""
    out = 0.0
    for a, n in enumerate(axes):
        k = 2.0 * math.pi * torch.fft.fftfreq(n, d=1.0 / n, dtype=torch.float64, device="cuda")
        out = out + (k ** 2).reshape([n if b == len(axes) - 1 - a else 1 for b in range(len(axes))])
    return out


def _position(axes, a):
    n = axes[a]
    x = torch.arange(n, dtype=torch.float64, device="cuda") / n
    return x.reshape([n if b == len(axes) - 1 - a else 1 for b in range(len(axes))])


def _classical(axes, n_tot, gen):
    """The classical field of the paper's test problem of that dimension, sum |psi|^2 dV = 1."""
    u = torch.rand(4, dtype=torch.float64, device="cuda", generator=gen).tolist()
    shape = tuple(reversed(axes))

    def soliton(center, rc):
        r2 = 0.0
        for a in range(len(axes)):
            d = _position(axes, a) - center[a]
            r2 = r2 + (d - torch.round(d)) ** 2
        return (1.0 + 0.091 * r2 / rc ** 2) ** -4

    if len(axes) == 1:       # a Gaussian overdensity
        x = _position(axes, 0)
        psi = torch.sqrt(1.0 + (0.4 + 0.2 * u[0]) * torch.exp(-(x - 0.4 - 0.2 * u[1]) ** 2 / (2 * 0.05 ** 2))) + 0j
    elif len(axes) == 2:     # two solitons moving toward each other
        k = 2.0 * math.pi / 0.1
        x, y = _position(axes, 0), 0.4 + 0.2 * u[0]
        psi = (soliton([0.35, y], 0.05) * torch.exp(1j * k * x)
               + soliton([0.65, y], 0.05) * torch.exp(-1j * k * x + 2j * math.pi * u[1]))
    elif n_tot >= 5e9:       # a stable collapsed object
        psi = soliton([0.4 + 0.2 * v for v in u[:3]], 1.0 / 16.0) + 0j
    else:                    # a Gaussian random field about to condense
        phase = torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen)
        psi = torch.fft.ifftn(torch.exp(-_k2(axes) / (2.0 * (16.0 * math.pi) ** 2) + 2j * math.pi * phase))
    dv = 1.0 / math.prod(axes)
    return (psi / torch.sqrt(torch.sum(torch.abs(psi) ** 2) * dv)).reshape(-1).contiguous()


def _batch(case, seed):
    """Classical field and streams of every instance, as the library lays a batch out."""
    gen, parts = _generator(seed), []
    for axes, streams in _instances(case):
        cl = _classical(axes, case["n_tot"], gen)
        cells = math.prod(axes)
        sigma = math.sqrt(0.5 * cells / (2.0 * case["n_tot"]))
        f = torch.empty((streams + 1, cells), dtype=torch.complex128 if case.get("f64") else torch.complex64, device="cuda")
        f[0] = cl
        for s in range(1, streams + 1):
            z = torch.randn((cells, 2), dtype=torch.float64, device="cuda", generator=gen)
            f[s] = cl + sigma * torch.view_as_complex(z)
        parts.append(f.reshape(-1))
    return parts[0] if len(parts) == 1 else torch.cat(parts)


def _weights(case, seed):
    """The surrogate's flat parameter vector, inputs and targets."""
    gen = _generator(seed)
    f32 = {"dtype": torch.float32, "device": "cuda", "generator": gen}
    w, n = case["width"], case["grid"]
    parts = [torch.randn(w * 4, **f32) * 0.5, torch.randn(w, **f32) * 0.1]
    for _ in range(case["layers"]):
        r = torch.rand((2 * case["modes"]) ** 3 * w * w * 2, **f32)
        parts += [r.mul_(2.0).sub_(1.0).div_(w), torch.randn(w * w, **f32) / math.sqrt(w), torch.randn(w, **f32) * 0.1]
    parts += [torch.randn(w, **f32) / math.sqrt(w), torch.randn(1, **f32) * 0.1]
    return (torch.cat(parts), torch.randn((case["batch"], 4, n, n, n), **f32),
            torch.randn((case["batch"], 1, n, n, n), **f32))


# ------------------------------------------------------------------------------- prepare, run, work
def prepare(case, seed):
    state = {"kind": case["kind"], "case": case}
    if case["kind"] in ("forward", "train"):
        theta, state["x"], state["t"] = _weights(case, seed)
        state["model"] = FNO(case["grid"], case["width"], case["modes"], case["layers"])
        state["model"].set_params(theta)
        return state
    hbar, dt = _physics(case)
    inst = _instances(case)
    ens = Ensemble([(len(a), a, 1.0) for a, _ in inst], hbar, COUPLING, dt, case["n_tot"], [s for _, s in inst],
                   precision=F64_PLAIN if case.get("f64") else F32)
    state["ens"] = ens
    if case["kind"] in ("sample", "run"):
        gen = _generator(seed)
        state["cl"] = torch.cat([_classical(a, case["n_tot"], gen) for a, _ in inst])
        state["seed"] = int(seed) * 2654435761 % 2 ** 63
    else:
        ens.psi.copy_(_batch(case, seed))
    if case["kind"] in ("run", "advance"):
        state["series"] = ens.new_series(case["steps"], case["every"])
    if case["kind"] == "phases":
        cells = math.prod(inst[0][0])
        state["out"] = [torch.empty(cells, dtype=torch.float64, device="cuda") for _ in range(2)]
    return state


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "forward":
        return state["model"].forward(state["x"])
    if kind == "train":
        loss = state["model"].train_step(state["x"], state["t"], 1e-4)
        return [loss, state["model"].get_params(0), state["model"].get_params(1)]
    ens = state["ens"]
    if kind == "sample":
        twa_sample(ens.h, state["cl"], state["seed"], ens.psi)
        return ens.psi
    if kind == "run":
        twa_run(ens.h, state["cl"], state["seed"], case["steps"], case["every"], ens.psi, state["series"])
        return [ens.psi, state["series"]]
    if kind == "advance":
        ens.advance(case["steps"], case["every"], state["series"])
        return [ens.psi, state["series"]]
    if kind == "step":
        ens.step(case["steps"])
        return ens.psi
    if kind == "dataset":
        ens.step(case["steps"])
        return [ens.psi] + [ens.moments(i) for i in range(len(ens.grids))]
    if kind == "moments":
        return ens.moments(0)
    return [*state["out"], twa_phase_moments(ens.h, 0, ens.psi, *state["out"])]


def work(case):
    if case["kind"] in ("forward", "train"):
        n3, w, b = case["grid"] ** 3, case["width"], case["batch"]
        m2, n = 2 * case["modes"], case["grid"]
        spectral = case["layers"] * m2 ** 3 * w * w * 2
        # per layer and direction: the truncated transform of w fields there and back, the mixing, the 1x1 map
        dft = 2 * w * (4.0 * n ** 3 * m2 + 8.0 * n * n * m2 * m2 + 8.0 * n * m2 ** 3)
        layer = b * (dft + 8.0 * m2 ** 3 * w * w + 2.0 * n3 * w * w)
        flops = case["layers"] * layer + b * 2.0 * n3 * w * 5
        if case["kind"] == "forward":
            return {"bytes": b * 5 * n3 * 4 + 2 * spectral, "flops": flops}
        # training also reads and writes the weights, both moments and the gradient, and returns two of them
        return {"bytes": b * 5 * n3 * 4 + (9 * 4 + 2) * spectral, "flops": 3.0 * flops}
    size = 16 if case.get("f64") else 8
    nbytes = flops = 0.0
    for axes, streams in _instances(case):
        cells, kind = math.prod(axes), case["kind"]
        values = (streams + 1) * cells
        fft = 5.0 * math.log2(cells)
        if kind == "sample":
            nbytes += values * size + 16 * cells
            flops += 60.0 * values
        elif kind in ("moments", "phases"):
            nbytes += values * size + 8 * cells * (7 if kind == "moments" else 2)
            flops += values * (fft + 20.0 if kind == "moments" else 30.0)
        else:
            nbytes += values * size * (1 if kind == "run" else 2)
            # two transforms of the field, two of its (real) density, the kick and the phase
            flops += case["steps"] * values * (3.0 * fft + 30.0)
            if kind == "dataset":
                nbytes += 8 * cells * 7
                flops += values * (fft + 20.0)
            elif kind != "step":
                flops += (case["steps"] // case["every"] + 1) * values * (fft + 20.0)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------------ in 64 bits
def _philox_normals(cells, slots, inst, seed):
    """Two standard normals a cell and slot: Philox4x32-10 words 0 and 1, Box-Muller."""
    mask = 0xFFFFFFFF
    c0 = torch.arange(cells, dtype=torch.int64, device="cuda")[None, :].expand(len(slots), cells)
    c1 = torch.tensor(slots, dtype=torch.int64, device="cuda")[:, None].expand(len(slots), cells)
    c2, c3 = torch.full_like(c0, inst), torch.zeros_like(c0)
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57     # products mod 2^64; the shifts below take their words
        c0, c1, c2, c3 = ((b >> 32) & mask) ^ c1 ^ k0, b & mask, ((a >> 32) & mask) ^ c3 ^ k1, a & mask
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    u0, u1 = (c0.double() + 0.5) / 2.0 ** 32, (c1.double() + 0.5) / 2.0 ** 32
    return torch.polar(torch.sqrt(-2.0 * torch.log(u0)), 2.0 * math.pi * u1)


def _exact_sample(case, seed):
    gen, out = _generator(seed), []
    key = int(seed) * 2654435761 % 2 ** 63
    inst = _instances(case)
    cls = [_classical(a, case["n_tot"], gen) for a, _ in inst]
    for i, (axes, streams) in enumerate(inst):
        cells = math.prod(axes)
        sigma = math.sqrt(0.5 * cells / (2.0 * case["n_tot"]))
        f = torch.empty((streams + 1, cells), dtype=torch.complex128, device="cuda")
        f[0] = cls[i]
        per = max(1, 2 ** 24 // cells)
        for s in range(1, streams + 1, per):
            slots = list(range(s, min(s + per, streams + 1)))
            f[s:s + len(slots)] = cls[i] + sigma * _philox_normals(cells, slots, i, key)
        out.append(f.reshape(-1))
    return torch.cat(out)


def _exact_steps(f, axes, hbar, dt, steps, every):
    """Steps the fields f (slots, cells) in place; yields them at the start and after every `every` steps."""
    shape, dims = tuple(reversed(axes)), tuple(range(1, len(axes) + 1))
    k2 = _k2(axes)
    drift = torch.polar(torch.ones_like(k2), -hbar * k2 * dt / 2.0)
    half = k2[..., : axes[0] // 2 + 1]
    poisson = torch.where(half > 0, -COUPLING / half, torch.zeros_like(half))
    g = f.reshape((-1,) + shape)

    def kick(frac):
        rho = g.real ** 2 + g.imag ** 2
        v = torch.fft.irfftn(torch.fft.rfftn(rho, dim=dims) * poisson, s=shape, dim=dims)
        g.mul_(torch.polar(torch.ones_like(v), v * (-frac * dt / hbar)))

    yield 0
    for s in range(1, steps + 1):
        kick(0.5)
        g.copy_(torch.fft.ifftn(torch.fft.fftn(g, dim=dims).mul_(drift), dim=dims))
        kick(0.5)
        if s % every == 0:
            yield s // every


class _Sums:
    """Sums over the streams of one instance, filled a few slots at a time (slot 0 first)."""

    def __init__(self, axes, streams, n_tot, modes):
        self.axes, self.cells, self.streams, self.n_tot, self.modes = axes, math.prod(axes), streams, n_tot, modes
        self.m2 = self.mean = self.a2 = self.a4 = 0.0

    def add(self, f, first):
        q = f[1:] if first else f
        if first:
            self.cl = f[0].real ** 2 + f[0].imag ** 2
            self.nk_cl = self._amp2(f[:1])[0] if self.modes else None
        self.m2 = self.m2 + (q.real ** 2 + q.imag ** 2).sum(0)
        self.mean = self.mean + q.sum(0)
        if self.modes:
            a = self._amp2(q)
            self.a2, self.a4 = self.a2 + a.sum(0), self.a4 + (a ** 2).sum(0)

    def _amp2(self, q):
        dims = tuple(range(1, len(self.axes) + 1))
        a = torch.fft.fftn(q.reshape((-1,) + tuple(reversed(self.axes))), dim=dims).reshape(q.shape)
        return (a.real ** 2 + a.imag ** 2) * (self.n_tot / self.cells ** 2)

    def scalars(self):
        dv = 1.0 / self.cells
        m2, mean = self.m2 / self.streams, self.mean / self.streams
        rho = m2 - self.cells / (2.0 * self.n_tot)
        d, c = torch.linalg.norm(rho - self.cl), torch.linalg.norm(self.cl)
        mass = m2.sum() * dv
        q = (m2 - mean.real ** 2 - mean.imag ** 2).sum() * dv - self.cells / (2.0 * self.n_tot)
        # the unitary transform keeps the sum of |a_k|^2
        return torch.stack([q, d / c, mass, self.cl.sum() * dv, torch.zeros_like(q),
                            self.n_tot * mass - 0.5 * self.cells, d, c])

    def outputs(self):
        m2, mean = self.m2 / self.streams, self.mean / self.streams
        a2 = self.a2 / self.streams
        # Var n_k cancels to far less than its terms: held to its type alone
        return {"rho_mean": m2 - self.cells / (2.0 * self.n_tot), "psi_mean": torch.view_as_real(mean).reshape(-1),
                "rho_cl": self.cl, "scalars": self.scalars(), "nk_mean": a2 - 0.5, "nk_var": None, "nk_cl": self.nk_cl}


def _exact_fields(case, psi):
    """The library's calls on the batch psi (complex128, stepped in place), as run() returns them."""
    kind, (hbar, dt) = case["kind"], _physics(case)
    steps = case.get("steps", 0)
    every = case["every"] if kind in ("run", "advance") else max(1, steps)
    at, rows, moments = 0, [], []
    for axes, streams in _instances(case):
        cells = math.prod(axes)
        f = psi[at:at + (streams + 1) * cells].reshape(streams + 1, cells)
        at += f.numel()
        sums = [_Sums(axes, streams, case["n_tot"], kind in ("dataset", "moments")) for _ in range(steps // every + 1)]
        per = max(2, 2 ** 25 // cells)
        for s in range(0, streams + 1, per):
            for o in _exact_steps(f[s:s + per], axes, hbar, dt, steps, every):
                if kind in ("run", "advance") or (kind != "step" and o == len(sums) - 1):
                    sums[o].add(f[s:s + per], s == 0)
        if kind in ("run", "advance"):
            rows.append(torch.stack([t.scalars() for t in sums]))
        elif kind != "step":
            moments.append(sums[-1].outputs())
    if kind in ("run", "advance"):
        return [psi, torch.stack(rows, 1)]
    return psi if kind == "step" else moments[0] if kind == "moments" else [psi] + moments


def _exact_phases(case, psi):
    (axes, streams), = _instances(case)
    cells = math.prod(axes)
    f = psi.reshape(streams + 1, cells)[1:]
    mean = f.mean(0)
    amp = torch.abs(f)
    am, va = amp.mean(0), amp.var(0, unbiased=False)
    unit = torch.where(torch.abs(mean) > 0, mean / torch.abs(mean), torch.ones_like(mean))
    p2 = (torch.angle(f * unit.conj()) ** 2).mean(0)
    rho = (amp ** 2).mean(0) - cells / (2.0 * case["n_tot"])
    return [va, p2, torch.stack([(rho * va / am).sum(), (rho * p2).sum() / (math.pi ** 2 / 3.0)]) / cells]


def _exact_network(case, seed):
    theta, x, t = _weights(case, seed)
    w, n, m, b = case["width"], case["grid"], case["modes"], case["batch"]
    m2 = 2 * m
    train = case["kind"] == "train"
    master, at, shapes = theta.double(), 0, [(w, 4), (w,)]
    for _ in range(case["layers"]):
        shapes += [(m2, m2, m2, w, w, 2), (w, w), (w,)]
    used = []                                # matrices are used rounded to bfloat16, biases as they are
    for sh in shapes + [(1, w), (1,)]:
        part = theta[at:at + math.prod(sh)]
        at += part.numel()
        part = (part.bfloat16() if len(sh) > 1 else part).double().reshape(sh)
        used.append(part.requires_grad_(train))
    keep = torch.tensor([i if i < m else n - m2 + i for i in range(m2)], device="cuda")

    def mat(weight, v, bias):
        return torch.einsum("oc,bck->bok", weight, v) + bias[None, :, None]

    with torch.set_grad_enabled(train):
        h = mat(used[0], x.double().reshape(b, 4, -1), used[1])
        for layer in range(case["layers"]):
            r, wl, bl = used[2 + 3 * layer: 5 + 3 * layer]
            s = torch.fft.fftn(h.reshape(b, w, n, n, n), dim=(2, 3, 4), norm="ortho")
            s = s.index_select(2, keep).index_select(3, keep).index_select(4, keep)
            s = torch.einsum("zyxoc,bczyx->bozyx", torch.view_as_complex(r), s)
            for d in (2, 3, 4):
                shape = list(s.shape)
                shape[d] = n
                s = torch.zeros(shape, dtype=s.dtype, device="cuda").index_copy(d, keep, s)
            z = torch.fft.ifftn(s, dim=(2, 3, 4), norm="ortho").real.reshape(b, w, -1) + mat(wl, h, bl)
            h = torch.nn.functional.gelu(z) if layer + 1 < case["layers"] else z
        y = mat(used[-2], h, used[-1]).reshape(t.shape)
        if not train:
            return y
        loss = ((y - t.double()) ** 2).mean()
        grad = torch.cat([g.reshape(-1) for g in torch.autograd.grad(loss, used)])
    # the first AdamW step from zero moments: the bias-corrected moments are the gradient and its square
    new = master - 1e-4 * (grad / (grad.abs() + 1e-8) + 1e-4 * master)
    return [loss.detach().reshape(1), new, grad]


def exact(case, seed):
    if case["kind"] in ("forward", "train"):
        return _exact_network(case, seed)
    if case["kind"] == "sample":
        return _exact_sample(case, seed)
    if case["kind"] == "run":
        # the run begins with the sampled batch rounded to the fields' 32 bits
        return _exact_fields(case, _exact_sample(case, seed).to(torch.complex64).to(torch.complex128))
    psi = _batch(case, seed).to(torch.complex128)
    return _exact_phases(case, psi) if case["kind"] == "phases" else _exact_fields(case, psi)
