"""The work that users of this framework have it do, as timed cases.

A case is a dict of plain values.  Its ``kind`` names the entry point:

* ``grid``    -- ``fft3d(x)``: complex grids through the functional call.
* ``plan``    -- ``Plan.execute``: a batch of orbitals, FP32 or a tensor-core
  kind, cubic or not.
* ``mixed``   -- ``MixedPlan.execute``: grids of different edges, forward,
  then the unnormalised inverse of the result.
* ``real``    -- ``rfft3d`` and ``irfft3d``: real grids to half spectra and
  back.
* ``hartree`` -- ``hartree_energy`` and its gradient through autograd.

Inputs are periodic complex Gaussians plus a little noise (localised
orbitals) or normalised real Gaussians holding 128 electrons (densities), as
in the package's ``synth`` module, made on the GPU from the seed.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2006_08435_gb300 import MixedPlan, Plan, fft3d, hartree_energy, irfft3d, rfft3d, synth

CELL = 10.0  # bohr
FUSED = (16, 32, 48, 64, 80, 96, 128)
# Edges of plane-wave grids: products of 2, 3 and 5.
SMOOTH = sorted(2 ** a * 3 ** b * 5 ** c for a in range(9) for b in range(6) for c in range(4)
                if 12 <= 2 ** a * 3 ** b * 5 ** c <= 320)
MAX_POINTS = 1 << 26  # complex points of the largest batches


def listed():
    return [
        # One grid of the paper's Table 1 per call: an SCF loop that works on
        # one orbital at a time.  Latency counts.
        dict(name="one_64", kind="grid", nx=64, ny=64, nz=64, batch=1, inverse=False, norm="none"),
        # One density's Hartree energy and potential per SCF step.
        dict(name="hartree_128_one", kind="hartree", n=128, batch=1),
        # All orbitals of a small system to reciprocal space: the two batches
        # of the benchmark's metric.
        dict(name="orbitals_64", kind="plan", nx=64, ny=64, nz=64, batch=256, precision="fp32",
             inverse=False, norm="none"),
        dict(name="orbitals_128", kind="plan", nx=128, ny=128, nz=128, batch=32, precision="fp32",
             inverse=False, norm="none"),
        # The same batch on the tensor cores.
        dict(name="orbitals_128_split", kind="plan", nx=128, ny=128, nz=128, batch=32,
             precision="split_fp16", inverse=False, norm="none"),
        # Back to real space, scaled, on a mixed-radix edge with a fused kernel.
        dict(name="orbitals_96_inv", kind="plan", nx=96, ny=96, nz=96, batch=48, precision="fp32",
             inverse=True, norm="by_n"),
        # Edges the cutoff dictates rather than the tuner: 2^2 5^2, a
        # non-cubic cell, and a large power of two.
        dict(name="cutoff_100_inv", kind="plan", nx=100, ny=100, nz=100, batch=16,
             precision="fp32", inverse=True, norm="none"),
        dict(name="cell_96x128x64", kind="plan", nx=96, ny=128, nz=64, batch=64, precision="fp32",
             inverse=False, norm="none"),
        dict(name="large_256", kind="plan", nx=256, ny=256, nz=256, batch=4, precision="fp32",
             inverse=False, norm="none"),
        # Real densities to half spectra and back, at an edge whose cell is
        # neither of the benchmark's two.
        dict(name="real_96", kind="real", n=96, batch=32),
        # Energies and gradients of a batch of densities (forward and backward).
        dict(name="hartree_128", kind="hartree", n=128, batch=32),
        # Grids of uneven cutoffs in one call, there and back.
        dict(name="mixed_64", kind="mixed", count=64, sizes_seed=0),
    ]


def _log_batch(rng: random.Random, points: int, limit: int, cap: int = 4096) -> int:
    most = max(1, min(cap, limit // points))
    return max(1, min(most, round(math.exp(rng.uniform(0.0, math.log(most + 0.5))))))


def draw(rng: random.Random):
    kind = rng.choice(["grid", "plan", "plan", "general", "general", "real", "hartree", "mixed"])
    norm = rng.choice(["none", "none", "by_n", "ortho"])
    inverse = rng.random() < 0.5
    if kind == "mixed":
        return dict(kind="mixed", count=rng.randint(4, 64), sizes_seed=rng.randint(0, 10 ** 6))
    if kind == "general":  # any box of plannable edges
        while True:
            e = [rng.choice(SMOOTH) for _ in range(3)]
            if rng.random() < 0.4:
                e = [e[0]] * 3
            pts = e[0] * e[1] * e[2]
            if pts <= MAX_POINTS // 2 and not (e[0] == e[1] == e[2] and e[0] in FUSED):
                break
        return dict(kind="plan", nx=e[0], ny=e[1], nz=e[2],
                    batch=_log_batch(rng, pts, MAX_POINTS // 2), precision="fp32",
                    inverse=inverse, norm=norm)
    if kind in ("grid", "plan"):
        precision = "fp32"
        if kind == "plan" and rng.random() < 0.25:
            precision = "split_fp16"
        n = rng.choice((64, 128) if precision != "fp32" else FUSED)
        c = dict(kind=kind, nx=n, ny=n, nz=n, batch=_log_batch(rng, n ** 3, MAX_POINTS),
                 inverse=inverse, norm=norm)
        if kind == "plan":
            c["precision"] = precision
        return c
    # real densities: even edges, a fused one half of the time
    n = rng.choice(FUSED) if rng.random() < 0.5 else rng.choice([s for s in SMOOTH
                                                                if s % 2 == 0 and s <= 216])
    return dict(kind=kind, n=n, batch=_log_batch(rng, n ** 3, MAX_POINTS // 3))


# ------------------------------------------------------------------ inputs
def _gauss_1d(n: int, centre, sigma, period: float, dev):
    """(count, n): periodic Gaussians on n points of one axis of length
    `period`, the nearest three images."""
    x = torch.arange(n, device=dev, dtype=torch.float64) * (period / n)
    d = x[None, :] - centre[:, None]
    acc = 0.0
    for m in (-1.0, 0.0, 1.0):
        acc = acc + torch.exp(-0.5 * ((d - m * period) / sigma[:, None]) ** 2)
    return acc


def _orbital(shape, gen, dev):
    """One complex64 grid: 8 Gaussians of width 0.5 .. 2 points with random
    phases, plus noise of 1e-3."""
    nz, ny, nx = shape
    u = torch.rand(8, 6, generator=gen, device=dev, dtype=torch.float64)
    sigma = 0.5 + 1.5 * u[:, 3]
    ax = [_gauss_1d(n, u[:, i] * n, sigma, float(n), dev) for i, n in enumerate((nx, ny, nz))]
    amp = torch.polar(0.5 + 0.5 * u[:, 4], 2 * math.pi * u[:, 5])
    gz = (ax[2] * amp[:, None]).to(torch.complex64)
    gy, gx = ax[1].to(torch.complex64), ax[0].to(torch.complex64)
    g = (gz.t() @ (gy[:, :, None] * gx[:, None, :]).reshape(8, ny * nx)).reshape(shape)
    noise = torch.rand(nz, ny, nx, 2, generator=gen, device=dev)
    return g + torch.view_as_complex(noise.mul_(2e-3).sub_(1e-3))


def _orbitals(shape, batch: int, seed: int):
    """A packed complex64 batch; at most 16 distinct orbitals, each repeat
    with a phase of its own."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)
    x = torch.empty((batch,) + tuple(shape), dtype=torch.complex64, device=dev)
    for b in range(batch):
        if b < 16:
            x[b] = _orbital(shape, gen, dev)
        else:
            t = 0.37 * b
            torch.mul(x[b % 16], complex(math.cos(t), math.sin(t)), out=x[b])
    return x


def _densities(n: int, batch: int, seed: int):
    """Real float32 densities of 128 electrons in a 10 bohr cell: 64
    normalised Gaussians each; at most 16 distinct, repeats shifted."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)
    rho = torch.empty((batch, n, n, n), dtype=torch.float32, device=dev)
    for b in range(batch):
        if b >= 16:
            rho[b] = torch.roll(rho[b % 16], shifts=b // 16, dims=0)
            continue
        u = torch.rand(64, 5, generator=gen, device=dev, dtype=torch.float64)
        sigma = 0.3 + 0.7 * u[:, 3]
        w = (1.0 - u[:, 4])
        w = w * (128.0 / w.sum()) * (2.0 * math.pi * sigma ** 2) ** -1.5
        gx, gy, gz = (_gauss_1d(n, u[:, i] * CELL, sigma, CELL, dev) for i in range(3))
        plane = (gy[:, :, None] * gx[:, None, :]).reshape(64, n * n)
        rho[b] = ((gz * w[:, None]).t() @ plane).reshape(n, n, n)
    return rho


def _mixed_input(dims, seed: int):
    parts = [_orbitals((n, n, n), 1, seed * 4099 + g).reshape(-1) for g, n in enumerate(dims)]
    return torch.cat(parts)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "grid":
        x = _orbitals((case["nz"], case["ny"], case["nx"]), case["batch"], seed)
        return dict(case=case, x=x)
    if kind == "plan":
        x = _orbitals((case["nz"], case["ny"], case["nx"]), case["batch"], seed)
        plan = Plan(case["nx"], case["ny"], case["nz"], case["batch"],
                    precision=case["precision"], inverse=case["inverse"], norm=case["norm"])
        return dict(case=case, x=x, plan=plan, out=torch.empty_like(x))
    if kind == "mixed":
        dims = synth.mixed_sizes(case["count"], seed=case["sizes_seed"])
        x = _mixed_input(dims, seed)
        return dict(case=case, x=x, fwd=MixedPlan(dims), inv=MixedPlan(dims, inverse=True),
                    mid=torch.empty_like(x), out=torch.empty_like(x))
    rho = _densities(case["n"], case["batch"], seed)
    if kind == "real":
        return dict(case=case, x=rho)
    ones = torch.ones(case["batch"], dtype=torch.float64, device=rho.device)
    return dict(case=case, x=rho.requires_grad_(True), ones=ones)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "grid":
        return fft3d(state["x"], inverse=case["inverse"], norm=case["norm"])
    if kind == "plan":
        return state["plan"].execute(state["x"], state["out"])
    if kind == "mixed":
        state["fwd"].execute(state["x"], state["mid"])
        state["inv"].execute(state["mid"], state["out"])
        return state["mid"], state["out"]
    if kind == "real":
        spec = rfft3d(state["x"])
        return spec, irfft3d(spec, norm="by_n")
    energy = hartree_energy(state["x"], CELL)
    (grad,) = torch.autograd.grad(energy, state["x"], grad_outputs=state["ones"])
    return energy.detach(), grad


def work(case):
    """One read of each input and one write of each output; 5 N log2 N
    operations for a complex transform of N points, half for a real one."""
    kind = case["kind"]
    if kind in ("grid", "plan"):
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 16 * n * case["batch"], "flops": 5 * n * math.log2(n) * case["batch"]}
    if kind == "mixed":
        pts = [n ** 3 for n in synth.mixed_sizes(case["count"], seed=case["sizes_seed"])]
        return {"bytes": 2 * 16 * sum(pts), "flops": 2 * sum(5 * p * math.log2(p) for p in pts)}
    n, b = case["n"], case["batch"]
    half = n * n * (n // 2 + 1)
    flops = 2 * 2.5 * n ** 3 * math.log2(n ** 3) * b
    if kind == "real":
        # the spectrum is an output of one call and an input of the next
        return {"bytes": (2 * 4 * n ** 3 + 2 * 8 * half) * b, "flops": flops}
    # the energy needs the whole spectrum of a density before the gradient
    # can start, but on-chip or not is the implementation's choice
    return {"bytes": (2 * 4 * n ** 3) * b + 8 * b, "flops": flops + 6 * half * b}


# ------------------------------------------------------------------- exact
def _scale(norm: str, n: int) -> float:
    return {"none": 1.0, "by_n": 1.0 / n, "ortho": 1.0 / math.sqrt(n)}[norm]


def _dft(x, inverse: bool, norm: str):
    """Eq. 1 of the paper over the last three axes, in FP64."""
    n = x.shape[-1] * x.shape[-2] * x.shape[-3]
    x = x.to(torch.complex128)
    if inverse:
        y = torch.fft.ifftn(x, dim=(-3, -2, -1), norm="forward")
    else:
        y = torch.fft.fftn(x, dim=(-3, -2, -1), norm="backward")
    return y.mul_(_scale(norm, n))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("grid", "plan"):
        x = _orbitals((case["nz"], case["ny"], case["nx"]), case["batch"], seed)
        return _dft(x, case["inverse"], case["norm"])
    if kind == "mixed":
        dims = synth.mixed_sizes(case["count"], seed=case["sizes_seed"])
        x = _mixed_input(dims, seed)
        parts = x.split([n ** 3 for n in dims])
        mid = torch.cat([_dft(p.reshape(n, n, n), False, "none").reshape(-1)
                         for p, n in zip(parts, dims)])
        return mid, torch.cat([p.to(torch.complex128) * n ** 3 for p, n in zip(parts, dims)])
    rho = _densities(case["n"], case["batch"], seed)
    n = case["n"]
    spec = torch.fft.rfftn(rho.double(), dim=(-3, -2, -1))
    if kind == "real":
        return spec, rho.double()
    m = torch.fft.fftfreq(n, 1.0 / n, device=rho.device, dtype=torch.float64)
    mx = torch.arange(n // 2 + 1, device=rho.device, dtype=torch.float64)
    m2 = m[:, None, None] ** 2 + m[None, :, None] ** 2 + mx[None, None, :] ** 2
    m2[0, 0, 0] = 1.0
    s = CELL ** 3 * 4.0 * math.pi / (float(n) ** 6 * (2.0 * math.pi / CELL) ** 2)
    wgt = torch.full((n // 2 + 1,), 2.0, device=rho.device, dtype=torch.float64)
    wgt[0] = wgt[-1] = 1.0
    k = wgt / m2
    k[0, 0, 0] = 0.0
    energy = 0.5 * s * ((spec.real ** 2 + spec.imag ** 2) * k).sum(dim=(-3, -2, -1))
    seed_spec = spec * (s / m2)
    seed_spec[:, 0, 0, 0] = 0.0
    grad = torch.fft.irfftn(seed_spec, s=(n, n, n), dim=(-3, -2, -1), norm="forward")
    return energy, grad
