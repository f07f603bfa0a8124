"""The work a user has this framework do, as measurable cases: whole calls through `fdtd.Context` and the
gradient drivers of `adjoint`, each pass one solve (or one gradient) from a state the program holds.

Kinds of cases:
  energy      FP64 vacuum PEC box with the discrete-energy record (the smallest solve users run: a
              conservation check of a new set-up)
  forward     one absorbing box of blocky permittivity, sheet source, spectra on the mid-plane
  cohort      several small absorbing boxes in one context (parameter sweeps)
  poles       several uneven two-pole Lorentz boxes in one context
  unitcell    a metasurface unit cell, periodic in x and y, absorbing in z, a flux monitor and a plane monitor
  gradient    checkpointed gradient of a spectral objective over a per-cell design box
  layer       the same with diagonal permittivity, a two-pole design layer, pole-parameter gradients and
              (by choice) BF16 snapshots
  reversible  the gradient of a lossless box by backward reconstruction
  streamed    the gradient of a box whose state lives in host memory
A pass is as long as the graph batches and remainders of a real run need to show, not as long as a full solve.
Forward cases continue from a developed field (a snapshot the program holds, restored in each pass).
"""
import math

import numpy as np
import torch

from paper_2609_30039_gb300 import adjoint as A
from paper_2609_30039_gb300 import fdtd as F
from paper_2609_30039_gb300 import workloads as W

START = 1000          # snapshot slot of the state a pass starts from (the replay uses the slots below)
DEV = "cuda:0"


def listed():
    return [
        # the smallest call: FP64 vacuum box, six fields and the energy of every step
        {"name": "energy_32_f64", "kind": "energy", "nx": 32, "ny": 32, "nz": 32, "steps": 200, "dtype": "f64"},
        # a sweep over eight small structures in one context
        {"name": "cohort_8x32", "kind": "cohort", "domains": 8, "nx": 32, "ny": 32, "nz": 32, "d": 6, "steps": 200,
         "dtype": "f32"},
        # the headline box: 128^3, 10-cell CPML, spectra of six components on a plane
        {"name": "forward_128", "kind": "forward", "nx": 128, "ny": 128, "nz": 128, "d": 10, "steps": 200,
         "dtype": "f32"},
        # the same box in FP64, the precision users check results with
        {"name": "forward_128_f64", "kind": "forward", "nx": 128, "ny": 128, "nz": 128, "d": 10, "steps": 64,
         "dtype": "f64"},
        # an ordinary box whose edges come from a geometry, not from a power of two
        {"name": "forward_ragged", "kind": "forward", "nx": 243, "ny": 251, "nz": 229, "d": 10, "steps": 101,
         "dtype": "f32"},
        # a large box: state far beyond the L2
        {"name": "forward_512", "kind": "forward", "nx": 512, "ny": 512, "nz": 512, "d": 10, "steps": 40,
         "dtype": "f32"},
        # uneven dispersive domains in one launch
        {"name": "lorentz_16", "kind": "poles", "domains": 16, "sizes": 1, "d": 8, "steps": 96, "dtype": "f32"},
        # a metasurface unit cell
        {"name": "unitcell", "kind": "unitcell", "nx": 96, "ny": 80, "nz": 200, "d": 10, "steps": 200, "dtype": "f32"},
        # inverse design: per-cell density box, binomial checkpoints
        {"name": "gradient_256", "kind": "gradient", "nx": 256, "ny": 256, "nz": 256, "d": 12, "steps": 64, "slots": 8,
         "dtype": "f32"},
        # anisotropic dispersive layer with compressed snapshots
        {"name": "layer_bf16", "kind": "layer", "nx": 128, "ny": 128, "nz": 128, "d": 16, "steps": 48, "slots": 6,
         "bf16": True, "dtype": "f32"},
        # lossless box, no checkpoints
        {"name": "reversible_128", "kind": "reversible", "nx": 128, "ny": 128, "nz": 128, "d": 0, "steps": 64,
         "dtype": "f32"},
        # a box stepped out of host memory
        {"name": "streamed_256", "kind": "streamed", "nx": 256, "ny": 256, "nz": 256, "d": 10, "steps": 16, "slab": 64,
         "halo": 8, "dtype": "f32"},
    ]


def _edge(rng, lo, hi):
    """A grid edge, spread over the logarithm of its range, of any residue."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["energy", "cohort", "forward", "forward", "forward", "forward", "poles", "unitcell", "gradient",
                       "layer", "reversible", "streamed"])
    c = {"kind": kind, "dtype": "f32"}
    if kind == "energy":
        return {**c, **{a: _edge(rng, 24, 64) for a in ("nx", "ny", "nz")}, "steps": rng.randint(100, 300),
                "dtype": "f64"}
    if kind == "cohort":
        n = rng.randint(24, 48)
        return {**c, "domains": rng.randint(2, 24), "nx": n, "ny": n, "nz": n, "d": rng.randint(4, 8),
                "steps": rng.randint(100, 300)}
    if kind == "forward":
        f64 = rng.random() < 0.25
        n = [_edge(rng, 48, 160 if f64 else 448) for _ in range(3)]
        if rng.random() < 0.5:   # half of the boxes have edges that are multiples of 8
            n = [8 * max(1, v // 8) for v in n]
        cells = n[0] * n[1] * n[2]
        steps = max(20, min(rng.randint(60, 260), int((5e8 if f64 else 3e9) / cells)))
        return {**c, "nx": n[0], "ny": n[1], "nz": n[2], "d": rng.randint(6, 12), "steps": steps,
                "dtype": "f64" if f64 else "f32"}
    if kind == "poles":
        return {**c, "domains": rng.randint(4, 24), "sizes": rng.randint(2, 1 << 30), "d": 8,
                "steps": rng.randint(60, 150)}
    if kind == "unitcell":
        return {**c, "nx": _edge(rng, 20, 160), "ny": _edge(rng, 20, 160), "nz": _edge(rng, 120, 320),
                "d": rng.randint(8, 12), "steps": rng.randint(100, 300)}
    if kind == "streamed":
        return {**c, **{a: _edge(rng, 128, 256) for a in ("nx", "ny", "nz")}, "d": rng.randint(8, 12),
                "steps": rng.randint(8, 16), "slab": rng.randint(40, 64), "halo": rng.randint(4, 8)}
    if kind == "reversible":
        return {**c, **{a: _edge(rng, 64, 200) for a in ("nx", "ny", "nz")}, "d": 0, "steps": rng.randint(32, 96)}
    top = 256 if kind == "gradient" else 144
    c = {**c, **{a: _edge(rng, 80, top) for a in ("nx", "ny", "nz")}, "d": rng.randint(8, 14),
         "steps": rng.randint(32, 64), "slots": rng.randint(5, 9)}
    return {**c, "bf16": rng.random() < 0.5} if kind == "layer" else c


# ------------------------------------------------------------------------------------- inputs
def _rng(seed, salt=0):
    return np.random.Generator(np.random.PCG64(7000003 * (int(seed) + 1) + salt))


def _blocks(rng, shape, lo, hi, low, high, block=8):
    """1 / eps: blocks of eps ~ U[low, high] in the box [lo, hi), 1 elsewhere; (nz, ny, nx) float32."""
    nx, ny, nz = shape
    inv = np.ones((nz, ny, nx), dtype=np.float32)
    ext = [h - l for l, h in zip(lo, hi)]
    b = (1.0 / rng.uniform(low, high, size=[-(-e // block) for e in reversed(ext)])).astype(np.float32)
    for ax in range(3):
        b = np.repeat(b, block, ax)
    inv[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]] = b[:ext[2], :ext[1], :ext[0]]
    return inv


def _pulse(rng, steps):
    """A pulse of about 20 cells' wavelength that peaks inside a short run."""
    return W.gaussian_pulse(steps, wavelength=float(rng.uniform(16.0, 24.0)), periods=0.5, delay=1.0)


OMEGAS = W.omegas_for((18.0, 20.0, 22.0))


def _box(case, rng, name, low=1.0, high=12.0):
    """Absorbing box, blocks of eps in its central half, Ez sheet near the low x face, six spectra on the z mid-plane."""
    n, d, steps = (case["nx"], case["ny"], case["nz"]), case["d"], case["steps"]
    inv = _blocks(rng, n, [v // 4 for v in n], [v - v // 4 for v in n], low, high)
    src = W.Source(W.EZ, (d + 5, d, d), (d + 6, n[1] - d, n[2] - d), _pulse(rng, steps))
    mon = W.Monitor((0, 0, n[2] // 2), (n[0], n[1], n[2] // 2 + 1), tuple(range(6)), OMEGAS)
    return W.Scene(shape=n, n_steps=steps, cpml=(d,) * 6, kappa_max=5.0, alpha_max=0.05, inv_eps=[inv], sources=[src],
                   monitors=[mon], name=name)


def _patch(n, d, z, comp, omegas=OMEGAS):
    c, hw = [v // 2 for v in n], [max(2, v // 32) for v in n]
    return W.Monitor((c[0] - hw[0], c[1] - hw[1], z), (c[0] + hw[0], c[1] + hw[1], z + 1), (comp,), omegas)


def _sizes(case):
    """Grids of a batch of uneven domains: every edge a multiple of 8 from 48 to 96."""
    rng = _rng(case["sizes"], 5)
    return [tuple(int(v) for v in 8 * rng.integers(6, 13, size=3)) for _ in range(case["domains"])]


def _half(case, n, rng):
    """The half-space of one axis, outside the absorbing faces, that a batch domain's poles fill: slices (z, y, x)."""
    d, axis = case["d"], int(rng.integers(0, 3))
    lo = [d] * 3
    lo[axis] = max(d, n[axis] // 2)
    return tuple(slice(lo[q], n[q] - d) for q in (2, 1, 0))


def _lorentz(case, n, rng):
    """A domain of a batch: two Lorentz poles (eps_inf 2) in a half-space, a point source, a point monitor."""
    d, steps = case["d"], case["steps"]
    half = _half(case, n, _rng(case["sizes"], sum(n)))
    mask = np.zeros(n[::-1], dtype=np.uint8)
    mask[half] = 1
    inv = np.ones(n[::-1], dtype=np.float32)
    inv[half] = 0.5
    poles = tuple((W.LORENTZ, float(rng.uniform(0.5, 3.0)), float(rng.uniform(0.05, 0.3)),
                   float(rng.uniform(0.001, 0.02))) for _ in range(2))
    p, m = [[int(rng.integers(d + 2, v - d - 2)) for v in n] for _ in range(2)]
    src = W.Source(W.EZ, tuple(p), tuple(v + 1 for v in p), _pulse(rng, steps))
    mon = W.Monitor(tuple(m), tuple(v + 1 for v in m), (W.EZ, W.HX), OMEGAS)
    return W.Scene(shape=n, n_steps=steps, cpml=(d,) * 6, kappa_max=5.0, alpha_max=0.05, inv_eps=[inv], poles=poles,
                   pole_mask=mask, sources=[src], monitors=[mon], name=case["kind"])


def _scenes(case, seed):
    kind, rng = case["kind"], _rng(seed)
    steps = case["steps"]
    if kind == "energy":
        n = (case["nx"], case["ny"], case["nz"])
        at = [int(rng.integers(v // 4, v - v // 4)) for v in n]
        wave = W.gaussian_derivative(steps, t0=float(rng.uniform(25, 35)), spread=float(rng.uniform(8, 12)))
        return [W.Scene(shape=n, n_steps=steps, name=kind, energy=True,
                        sources=[W.Source(W.EZ, tuple(at), tuple(v + 1 for v in at), wave)])]
    if kind == "cohort":
        return [_box(case, _rng(seed, 1 + q), kind) for q in range(case["domains"])]
    if kind == "poles":
        return [_lorentz(case, n, _rng(seed, 1 + q)) for q, n in enumerate(_sizes(case))]
    n = (case["nx"], case["ny"], case["nz"])
    if kind == "forward":
        return [_box(case, rng, kind)]
    d = case["d"]
    if kind == "streamed":
        sc = _box(case, rng, kind)
        q = [(v // 2 - v // 16, v // 2 + v // 16) for v in n]
        sc.design = (tuple(a for a, _ in q), tuple(b for _, b in q))
        c = [v // 2 for v in n]
        sc.sources = [W.Source(W.EZ, (c[0], c[1], d), (c[0] + 1, c[1] + 1, n[2] - d), _pulse(rng, steps))]
        sc.monitors = [_patch(n, d, c[2], W.EZ)]
        return [sc]
    if kind == "unitcell":
        z = (2 * n[2] // 5, 3 * n[2] // 5)
        inv = np.ones((n[2], n[1], n[0]), dtype=np.float32)
        eps = rng.uniform(1.0, 6.0, size=(-(-n[1] // 4), -(-n[0] // 4)))
        inv[z[0]:z[1]] = (1.0 / np.repeat(np.repeat(eps, 4, 0), 4, 1)[:n[1], :n[0]]).astype(np.float32)
        src = W.Source(W.EX, (0, 0, d + 2), (n[0], n[1], d + 3), _pulse(rng, steps))
        flux = W.Monitor((0, 0, z[1] + 4), (n[0], n[1], z[1] + 6), (W.EX, W.EY, W.HX, W.HY), OMEGAS)
        plane = W.Monitor((0, 0, n[2] // 2), (n[0], n[1], n[2] // 2 + 1), tuple(range(6)), OMEGAS)
        return [W.Scene(shape=n, n_steps=steps, cpml=(0, 0, 0, 0, d, d), kappa_max=3.0, alpha_max=0.05, inv_eps=[inv],
                        sources=[src], monitors=[flux, plane], periodic=(1, 1, 0), name=kind)]
    if kind == "gradient":
        lo, hi = [n[0] // 4, n[1] // 4, (7 * n[2]) // 16], [n[0] - n[0] // 4, n[1] - n[1] // 4, (9 * n[2]) // 16]
        rho = rng.uniform(0.0, 1.0, size=[h - l for l, h in zip(reversed(lo), reversed(hi))])
        inv = np.ones((n[2], n[1], n[0]), dtype=np.float32)
        inv[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]] = 1.0 / W.density_to_eps(rho)
        src = W.Source(W.EX, (d, d, lo[2] - 4), (n[0] - d, n[1] - d, lo[2] - 3), _pulse(rng, steps))
        return [W.Scene(shape=n, n_steps=steps, cpml=(d,) * 6, kappa_max=5.0, alpha_max=0.05, inv_eps=[inv],
                        sources=[src], monitors=[_patch(n, d, hi[2] + 4, W.EX)], design=(tuple(lo), tuple(hi)),
                        rho=rho, name=kind)]
    if kind == "layer":
        m = d + 4
        inv = [_blocks(rng, n, [m] * 3, [v - m for v in n], 1.0, 6.0, block=4) for _ in range(3)]
        lo = [m, m, n[2] // 2 - max(2, n[2] // 20)]
        hi = [n[0] - m, n[1] - m, n[2] // 2 + max(2, n[2] // 20)]
        mask = np.zeros((n[2], n[1], n[0]), dtype=np.uint8)
        mask[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]] = 1
        poles = tuple((W.LORENTZ, float(rng.uniform(0.5, 3.0)), float(rng.uniform(0.05, 0.3)),
                       float(rng.uniform(0.001, 0.02))) for _ in range(2))
        src = W.Source(W.EY, (d, d, lo[2] - 6), (n[0] - d, n[1] - d, lo[2] - 5), _pulse(rng, steps))
        mon = W.Monitor((lo[0], lo[1], hi[2] + 4), (hi[0], hi[1], hi[2] + 5), (W.EY,), W.omegas_for((19.0, 21.0)))
        return [W.Scene(shape=n, n_steps=steps, cpml=(d,) * 6, kappa_max=5.0, alpha_max=0.05, inv_eps=inv, poles=poles,
                        pole_mask=mask, sources=[src], monitors=[mon], design=(tuple(lo), tuple(hi)), name=kind)]
    # reversible: lossless, periodic in x, the design box against the seam
    inv = _blocks(rng, n, [0, 0, 0], list(n), 1.0, 6.0)
    design = ((0, (3 * n[1]) // 8, (7 * n[2]) // 16), (n[0] // 8, (5 * n[1]) // 8, (9 * n[2]) // 16))
    src = W.Source(W.EZ, (0, 1, n[2] // 2 - 8), (n[0], n[1], n[2] // 2 - 7), _pulse(rng, steps))
    return [W.Scene(shape=n, n_steps=steps, cpml=(0,) * 6, inv_eps=[inv], sources=[src],
                    monitors=[W.Monitor((0, n[1] // 2 - 4, design[1][2] + 2), (8, n[1] // 2 + 4, design[1][2] + 3),
                                        (W.EX,), OMEGAS)],
                    design=design, periodic=(1, 0, 0), name=kind)]


def _warm(sc, seed, dtype):
    """A developed field: per component two standing waves of 10 to 40 cells (whole periods on a periodic axis,
    faded out towards the faces of the others, zero where a wall holds them); (6, nz, ny, nx) of `dtype`."""
    rng = _rng(seed, 977)
    out = torch.empty((6,) + sc.shape[::-1], dtype=dtype, device=DEV)
    for c in range(6):
        a = None
        for _ in range(2):
            f = []
            for q in range(3):
                N = sc.shape[q]
                x = torch.arange(N, dtype=torch.float64, device=DEV) + 0.5
                per, ph = rng.uniform(10.0, 40.0), rng.uniform(0.0, 2 * math.pi)
                if sc.periodic[q]:
                    f.append(torch.sin(2 * math.pi * x * max(1, round(N / per)) / N + ph))
                else:
                    f.append(torch.sin(2 * math.pi * x / per + ph) * torch.sin(math.pi * x / N) ** 2)
            f = [v.to(dtype) for v in f]
            t = 0.5 * f[2][:, None, None] * f[1][None, :, None] * f[0][None, None, :]
            a = t if a is None else a + t
        if c < 3:
            for q in range(3):
                if q != c and not sc.periodic[q]:
                    a.select(2 - q, 0).zero_()
        out[c] = a
    return out


# a run without a held state starts at rest: the energy record belongs to a whole run, and a host-streamed
# context keeps no snapshots
def _rest(case):
    return case["kind"] in ("energy", "streamed")


class State:
    pass


def prepare(case, seed):
    s = State()
    s.kind, s.steps = case["kind"], case["steps"]
    scs = _scenes(case, seed)
    s.ctx = F.Context(scs, dtype=case["dtype"],
                      streamed=(case["slab"], case["halo"]) if case["kind"] == "streamed" else None)
    s.rest = _rest(case)
    if not s.rest:
        for dom, sc in enumerate(scs):
            f = _warm(sc, int(seed) + 31 * dom, s.ctx.tdtype)
            for c in range(6):
                s.ctx.set_part(dom, c, f[c])
        F.fdtd_state_save(s.ctx.ctx, START, F.FDTD_CODEC_NATIVE)
    s.runner = None
    if case["kind"] in ("gradient", "layer"):
        s.runner = A.DesignAdjoint(s.ctx, slots=case["slots"],
                                   codec=F.FDTD_CODEC_BF16 if case.get("bf16") else F.FDTD_CODEC_NATIVE,
                                   pole_grads=case["kind"] == "layer")
    elif case["kind"] == "reversible":
        s.runner = A.ReversibleAdjoint(s.ctx)
    elif case["kind"] == "streamed":
        s.runner = A.StreamedAdjoint(s.ctx)
    return s


def _loss(specs):
    """J = sum |F|^2 over every monitor value, and its cotangents dJ/dRe F + i dJ/dIm F."""
    return float(sum((f.real.square() + f.imag.square()).sum() for f in specs)), [2.0 * f for f in specs]


def _field_precision(s, v):
    """Spectra and gradients are accumulated in FP64; a program of FP32 fields takes them on in FP32."""
    if s.ctx.tdtype == torch.float64:
        return v
    if isinstance(v, np.ndarray):
        return v.astype(np.float32)
    return v.to(torch.complex64 if v.is_complex() else torch.float32)


def run(s):
    c = s.ctx.ctx
    F.fdtd_reset(c) if s.rest else F.fdtd_state_restore(c, START)
    F.fdtd_dft_reset(c)
    out = {}
    if s.runner is not None:
        (J, specs), grads, _ = s.runner.run(s.steps, _loss)
        out = {"J": J, "spectra": _field_precision(s, specs[0]), "grad": _field_precision(s, grads[0])}
        if s.kind == "layer":
            out["pole_grad"] = _field_precision(s, s.runner.pole_grads[0])
        return out
    s.ctx.step(s.steps)
    if s.kind in ("cohort", "poles"):   # one tensor of every domain's fields, and one of all spectra
        nd = len(s.ctx.scenes)
        out["fields"] = torch.cat([s.ctx.part(d, q) for d in range(nd) for q in range(6)])
        out["spectra"] = _field_precision(s, torch.cat([s.ctx.dft(k).reshape(-1) for k in range(len(s.ctx.monitors))]))
        return out
    out["fields"] = [s.ctx.field(0, q) for q in range(6)]
    if s.kind == "energy":   # as one tensor: Hz of an Ez source in an empty box is nothing but rounding
        out["fields"] = torch.stack(out["fields"])
        out["energy"] = s.ctx.energy(0, s.steps)
    else:
        out["spectra"] = [_field_precision(s, s.ctx.dft(k)) for k in range(len(s.ctx.monitors))]
    if s.kind == "unitcell":
        out["flux"] = _field_precision(s, F.fdtd_dft_flux(c, s.ctx.monitors[0][0], len(OMEGAS)))
    return out


# ------------------------------------------------------------------------------------- what a pass needs
def work(case):
    """Per time step (forward, backward or transposed) the state of a cell is read once and written once: six
    fields in and out and 1/eps in; per CPML slab a cell lies in, the four memories of that axis in and out; two
    poles in a dispersive cell: 12 pole values in and out.  36 operations per cell (12 per slab membership, 8 per
    pole and component) beside them; per DFT sample and frequency 4.  A gradient needs its forward sweep, the
    replays its checkpoints leave to it, and the transposed steps; a host-streamed one its window replays."""
    w = 8 if case["dtype"] == "f64" else 4
    kind, steps = case["kind"], case["steps"]
    if kind == "poles":
        shapes = _sizes(case)
    else:
        shapes = [(case["nx"], case["ny"], case["nz"])] * case.get("domains", 1)
    d = case.get("d", 0)
    nbytes = flops = 0.0
    for n in shapes:
        cells = float(n[0] * n[1] * n[2])
        axes = [2] if kind == "unitcell" else [0, 1, 2] if d else []
        member = sum(2.0 * d / n[a] for a in axes) * cells
        iso = 3 if kind == "layer" else 1
        b = w * ((12 + iso) * cells + 8 * member)
        f = 36 * cells + 48 * member
        disp = 0.0
        if kind == "poles":
            disp = float(math.prod(v.stop - v.start for v in _half(case, n, _rng(case["sizes"], sum(n)))))
        elif kind == "layer":
            disp = float((n[0] - 2 * d - 8) * (n[1] - 2 * d - 8) * 2 * max(2, n[2] // 20))
        b += w * 24 * disp
        f += 48 * disp
        spec = {"forward": 6 * 3 * n[0] * n[1], "cohort": 6 * 3 * n[0] * n[1],
                "unitcell": 14 * 3 * n[0] * n[1]}.get(kind, 0)
        f += 4 * spec
        nbytes += b
        flops += f
    if kind in ("gradient", "layer"):
        st = A.replay_stats(A.schedule(steps, case["slots"]))
        passes = st["forward_steps"] + st["adjoint_steps"]
    elif kind == "reversible":
        passes = 3 * steps
    elif kind == "streamed":
        passes = 3 * steps
    else:
        passes = steps
    return {"bytes": nbytes * passes, "flops": flops * passes}


# ------------------------------------------------------------------------------------- the same in 64 bits
def _d(f, q, per, back):
    """Difference of a field (nz, ny, nx) along axis q: f(x) - f(x - 1) (back) or f(x + 1) - f(x); the absent
    neighbour beyond a wall is 0."""
    dim, n = 2 - q, f.shape[2 - q]
    if per:
        return f - torch.roll(f, 1, dim) if back else torch.roll(f, -1, dim) - f
    z = torch.zeros_like(f.narrow(dim, 0, 1))
    if back:
        return f - torch.cat([z, f.narrow(dim, 0, n - 1)], dim)
    return torch.cat([f.narrow(dim, 1, n - 1), z], dim) - f


def _profile(sc, q, half):
    """CPML rows b, c, 1/kappa over the two slabs of axis q (E at integer, H at half-integer nodes), low slab first."""
    N, lo, hi = sc.shape[q], sc.cpml[2 * q], sc.cpml[2 * q + 1]
    smax = 0.8 * (sc.cpml_m + 1.0) if sc.sigma_max < 0 else sc.sigma_max
    rows = np.zeros((3, N))
    for j in range(N):
        x = j + (0.5 if half else 0.0)
        rho, dep = (lo - x, lo) if lo and x < lo else (x - (N - hi), hi) if hi and x > N - hi else (-1.0, 1.0)
        rows[:, j] = 1.0, 0.0, 1.0
        if rho >= 0:
            r = min(rho / dep, 1.0)
            sig, kap, al = smax * r ** sc.cpml_m, 1 + (sc.kappa_max - 1) * r ** sc.cpml_m, sc.alpha_max * (1 - r)
            b = math.exp(-(sig / kap + al) * sc.courant)
            rows[:, j] = b, sig * (b - 1) / (sig * kap + kap * kap * al) if sig > 0 else 0.0, 1 / kap
    shape = [1, 1, 1]
    shape[2 - q] = lo + hi
    return [torch.tensor(np.concatenate([r[:lo], r[N - hi:]]), device=DEV).reshape(shape) for r in rows]


def _slabs(f, dim, lo, hi):
    return torch.cat([f.narrow(dim, 0, lo), f.narrow(dim, f.shape[dim] - hi, hi)], dim)


class _Model:
    """The scheme of one scene in plain 64-bit torch operations."""

    def __init__(self, sc, f0, ie, poles=None):
        self.sc, self.S = sc, sc.courant
        n = sc.shape[::-1]
        zero = lambda: torch.zeros(n, dtype=torch.float64, device=DEV)  # noqa: E731
        self.f = [v.to(torch.float64) for v in f0] if f0 is not None else [zero() for _ in range(6)]
        self.ie = ie
        self.prof = [[_profile(sc, q, h) if sc.cpml[2 * q] or sc.cpml[2 * q + 1] else None for q in range(3)]
                     for h in (False, True)]
        self.psi = {(c, s): 0.0 for c in range(6) for s in (0, 1)}
        self.free = []   # 1 on an E component's nodes that no wall holds
        for a in range(3):
            m = torch.ones(n, dtype=torch.float64, device=DEV)
            for q in range(3):
                if q != a and not sc.periodic[q]:
                    m.select(2 - q, 0).zero_()
            self.free.append(m)
        self.x, self.poles = {}, poles
        if poles is not None:
            self.mask = torch.tensor(sc.pole_mask, dtype=torch.float64, device=DEV)
            self.coef = [self._pole(k, *p) for (k, _, _, _), p in zip(sc.poles, poles)]
        self.n = 0
        self.acc = [torch.zeros((len(m.comps), len(m.omegas)) + tuple(h - l for l, h in zip(m.lo, m.hi))[::-1],
                                dtype=torch.complex128, device=DEV) for m in sc.monitors]
        self.energy = []

    @staticmethod
    def _pole(kind, deps, om, gam):
        a0 = om * om if kind == W.LORENTZ else 0.0 * om
        b1 = deps * om * om if kind == W.LORENTZ else om * om
        det = 1 + gam / 2 + a0 / 4
        return (1 + gam / 2 - a0 / 4) / det, 1 / det, -a0 / det, (1 - gam / 2 - a0 / 4) / det, b1 / (4 * det), b1 / (2 * det)

    def _curl(self, c, fields, half):
        """Both CPML-corrected derivatives of component c (an E one: of H, backwards; an H one: of E, forwards)."""
        a, out = c % 3, []
        for s in (0, 1):
            q, o = (a + 1 + s) % 3, (a + 2 - s) % 3
            D = _d(fields[o], q, self.sc.periodic[q], not half)
            p = self.prof[half][q]
            if p is not None:   # in the slabs: the memory advances, then D / kappa + memory
                lo, hi, dim = self.sc.cpml[2 * q], self.sc.cpml[2 * q + 1], 2 - q
                Ds = _slabs(D, dim, lo, hi)
                ps = p[0] * self.psi[c, s] + p[1] * Ds
                self.psi[c, s] = ps
                y = p[2] * Ds + ps
                D = torch.cat([y.narrow(dim, 0, lo), D.narrow(dim, lo, D.shape[dim] - lo - hi), y.narrow(dim, lo, hi)], dim)
            out.append(D)
        return out[0] - out[1]

    def _sources(self, f, lo, n):
        for src in self.sc.sources:
            if lo <= src.comp < lo + 3 and n < len(src.wave):
                f[src.comp] = f[src.comp].clone()
                f[src.comp][src.lo[2]:src.hi[2], src.lo[1]:src.hi[1], src.lo[0]:src.hi[0]] += float(src.wave[n])

    def _dft(self, f, lo, t):
        for m, acc in zip(self.sc.monitors, self.acc):
            for ci, c in enumerate(m.comps):
                if lo <= c < lo + 3:
                    v = f[c].detach()[m.lo[2]:m.hi[2], m.lo[1]:m.hi[1], m.lo[0]:m.hi[0]]
                    for k, w in enumerate(m.omegas):
                        acc[ci, k] += v * complex(math.cos(w * t), math.sin(w * t))

    def cotangents(self, cots, lo, t):
        """d J / d field of the samples taken at time t: [(component, box, value)]."""
        out = []
        for m, ct in zip(self.sc.monitors, cots):
            for ci, c in enumerate(m.comps):
                if lo <= c < lo + 3:
                    v = sum(ct[ci, k].real * math.cos(w * t) + ct[ci, k].imag * math.sin(w * t)
                            for k, w in enumerate(m.omegas))
                    out.append((c, (slice(m.lo[2], m.hi[2]), slice(m.lo[1], m.hi[1]), slice(m.lo[0], m.hi[0])), v))
        return out

    def step(self):
        f = list(self.f)
        n, S, H = self.n, self.S, self.f[3:]
        new = []
        for a in range(3):
            cu, e0 = self._curl(a, H, False), f[a]
            if self.poles is None:
                new.append(e0 + S * self.free[a] * (self.ie[a] * cu))
                continue
            G = sum(co[4] for co in self.coef) * self.mask
            delta = S * self.free[a] * cu
            for p, co in enumerate(self.coef):
                P, Q = self.x.get((a, p), (0.0, 0.0))
                delta = delta + (P - (co[0] * P + co[1] * Q) - 2 * co[4] * e0 * self.mask)
            e1 = e0 + self.ie[a] / (1 + self.ie[a] * G) * delta
            for p, co in enumerate(self.coef):
                P, Q = self.x.get((a, p), (0.0, 0.0))
                es = (e1 + e0) * self.mask
                self.x[a, p] = (co[0] * P + co[1] * Q + co[4] * es, co[2] * P + co[3] * Q + co[5] * es)
            new.append(e1)
        f[:3] = new
        self._sources(f, 0, n)
        self._dft(f, 0, n + 1)
        h0 = f[3:]
        f[3:] = [h0[a] - S * self._curl(3 + a, f[:3], True) for a in range(3)]
        if self.sc.energy:
            w = sum((e * e / i).sum() for e, i in zip(f[:3], self.ie)) + sum((x * y).sum() for x, y in zip(h0, f[3:]))
            self.energy.append(0.5 * float(w))
        self._sources(f, 3, n)
        self._dft(f, 3, n + 1.5)
        self.f, self.n = f, n + 1

    def state(self):
        """Every tensor the next step reads, as a flat list of (key, tensor)."""
        return ([(("f", c), self.f[c]) for c in range(6)] + [(("psi", k), v) for k, v in self.psi.items()] +
                [(("x", k + (w,)), v[w]) for k, v in self.x.items() for w in (0, 1)])

    def load(self, st, n):
        self.n = n
        self.f = [st["f", c] for c in range(6)]
        self.psi = {k: st["psi", k] for k in self.psi}
        keys = {k[1][:2] for k in st if k[0] == "x"}
        self.x = {k: (st["x", k + (0,)], st["x", k + (1,)]) for k in keys}


def _gradient(model, sc, leaves, steps):
    """J and dJ/dleaves, by autograd one step at a time from the kept states of the forward sweep."""
    kept = []
    with torch.no_grad():
        for _ in range(steps):
            kept.append([(k, v if not torch.is_tensor(v) else v.detach()) for k, v in model.state()])
            model.step()
    J, cots = _loss_exact(model.acc)
    bar = {}
    grads = [torch.zeros_like(v) for v in leaves[0]]
    mon, sc.monitors = sc.monitors, []          # the replayed steps take no spectra
    for n in reversed(range(steps)):
        sc.monitors = mon
        inj = model.cotangents(cots, 0, n + 1) + model.cotangents(cots, 3, n + 1.5)
        sc.monitors = []
        ins = {k: (v.requires_grad_() if torch.is_tensor(v) else v) for k, v in kept.pop()}
        vars_ = leaves[0]
        leaves[1](model)
        model.load(ins, n)
        model.step()
        outs = [(k, v) for k, v in model.state() if torch.is_tensor(v) and v.requires_grad]
        seed = []
        for k, v in outs:
            b = bar.get(k)
            b = torch.zeros_like(v) if b is None else b
            for c, box, val in inj:
                if k == ("f", c):
                    b = b.clone()
                    b[box] += val
            seed.append(b)
        wrt = [(k, v) for k, v in ins.items() if torch.is_tensor(v)]
        got = torch.autograd.grad([v for _, v in outs], [v for _, v in wrt] + list(vars_), seed, allow_unused=True)
        bar = {k: g for (k, _), g in zip(wrt, got) if g is not None}
        for t, g in zip(grads, got[len(wrt):]):
            if g is not None:
                t += g
        del outs, ins, wrt, got, seed
    sc.monitors = mon
    return J, grads


def _loss_exact(accs):
    return float(sum((f.real ** 2 + f.imag ** 2).sum() for f in accs)), [2 * f for f in accs]


def exact(case, seed):
    scs = _scenes(case, seed)
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    steps, kind, rest = case["steps"], case["kind"], _rest(case)
    models = []
    for dom, sc in enumerate(scs):
        f0 = None if rest else _warm(sc, int(seed) + 31 * dom, dt)
        arrs = sc.inv_eps3()
        ie = [torch.tensor(np.asarray(a), device=DEV).to(dt).double() for a in (arrs[:1] if arrs[0] is arrs[1] else arrs)]
        ie = ie * 3 if len(ie) == 1 else ie
        poles = None
        if len(sc.poles):
            poles = [[torch.tensor(float(v), dtype=torch.float64, device=DEV) for v in p[1:]] for p in sc.poles]
        if kind in ("gradient", "layer", "reversible", "streamed"):
            return _exact_gradient(case, sc, f0, ie, poles)
        m = _Model(sc, f0, ie, poles)
        with torch.no_grad():
            for _ in range(steps):
                m.step()
        models.append(m)
    if kind in ("cohort", "poles"):
        return {"fields": torch.cat([v.reshape(-1) for m in models for v in m.f]),
                "spectra": torch.cat([v.reshape(-1) for m in models for v in m.acc])}
    m = models[0]
    out = {"fields": torch.stack(m.f) if kind == "energy" else m.f}
    if kind == "energy":
        out["energy"] = np.array(m.energy)
    else:
        out["spectra"] = m.acc
    if kind == "unitcell":
        a = m.acc[0]   # components Ex, Ey, Hx, Hy on two planes
        ex, ey = (a[0][:, 0] + a[0][:, 1]) / 2, (a[1][:, 0] + a[1][:, 1]) / 2
        hx, hy = a[2][:, 0], a[3][:, 0]
        out["flux"] = (0.5 * (ex * hy.conj() - ey * hx.conj()).real.sum((1, 2))).cpu().numpy()
    return out


def _exact_gradient(case, sc, f0, ie, poles):
    (lx, ly, lz), (hx, hy, hz) = sc.design
    box = (slice(lz, hz), slice(ly, hy), slice(lx, hx))
    leaves = [torch.stack([i[box] for i in ie]).requires_grad_()]
    pl = [v.requires_grad_() for p in poles for v in p] if poles is not None else []
    model = _Model(sc, f0, ie, poles)

    def bind(m):
        m.ie = []
        for a in range(3):
            i = ie[a].clone()
            i[box] = leaves[0][a]
            m.ie.append(i)
        if poles is not None:
            m.coef = [m._pole(k, *p) for (k, _, _, _), p in zip(sc.poles, poles)]

    J, grads = _gradient(model, sc, (leaves + pl, bind), case["steps"])
    out = {"J": J, "spectra": model.acc[0], "grad": grads[0].reshape(-1)}
    if poles is not None:
        out["pole_grad"] = np.array([float(g) for g in grads[1:]]).reshape(-1, 3)
    return out
