"""Per-cell updates by groups of cells along x: every row length, slab depth and alignment that picks another group
length, or meets a group's edge, gives the bits of the tile launches (which update cell by cell)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2609_30039_gb300 import fdtd  # noqa: E402
from paper_2609_30039_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _scene(nx, cpml, periodic, n_iso, dtype, poles=False):
    ny, nz, n = 13, 11, 37
    rng = np.random.default_rng(nx * 100 + sum(cpml))
    inv = [np.ones((nz, ny, nx)) for _ in range(n_iso)]
    mid = tuple(slice(3, -3) for _ in range(2)) + (slice(cpml[0], nx - cpml[1]),)
    for a in inv:
        a[mid] = rng.uniform(0.2, 1.0, size=a[mid].shape)
    x = min(cpml[0] + 1, nx - 1)
    src = [W.Source(W.EZ, (x, 1, 2), (x + 1, ny, nz - 2), W.gaussian_pulse(n, 8.0, periods=0.5, delay=1.0)),
           W.Source(W.HX, (0, 2, 3), (nx, 5, 4), W.gaussian_pulse(n, 9.0, periods=0.5, delay=1.0)),
           W.Source(W.EX, (1, 4, 5), (min(nx, 6), 7, 6), W.gaussian_pulse(n, 7.0, periods=0.5, delay=1.0))]
    mon = W.Monitor((0, 1, 4), (nx, ny, 6), (W.EX, W.EZ, W.HY), W.omegas_for((8.0, 9.0)))
    mask = None
    if poles:
        mask = np.zeros((nz, ny, nx), dtype=np.uint8)
        mask[4:7, 3:10, cpml[0] + (nx % 3): nx - cpml[1] - 1] = 1
        mask[5, 5, :] = 0
    pl = tuple((W.LORENTZ, 1.0 + p, 0.1 + 0.05 * p, 0.01) for p in range(poles))
    return W.Scene(shape=(nx, ny, nz), n_steps=n, cpml=cpml, kappa_max=3.0, alpha_max=0.05, inv_eps=inv, sources=src,
                   monitors=[mon], periodic=periodic, poles=pl, pole_mask=mask)


def _run(sc, dtype, mode, shift=0):
    ctx = fdtd.Context(sc, dtype=dtype)
    fdtd.fdtd_set_launch_mode(ctx.ctx, mode)
    if shift:   # the caller's eps^-1 off its 16-byte boundary
        ie = []
        for t in ctx.inv_eps[0]:
            buf = torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)
            buf[shift:] = t.reshape(-1)
            ie.append(buf[shift:].view(t.shape))
        ctx.set_inv_eps(0, ie)
    ctx.step(35)
    ctx.step(2)
    out = [ctx.part(0, p).clone() for p in range(ctx.part_count(0))] + [ctx.dft(0).clone()]
    ctx.close()
    return out


@pytest.mark.parametrize("nx,cpml,periodic", [
    (2, (0, 0, 2, 2, 2, 2), (0, 0, 0)), (4, (0, 0, 2, 2, 0, 3), (1, 0, 0)), (7, (2, 3, 0, 2, 2, 0), (0, 0, 0)),
    (8, (3, 3, 2, 2, 2, 2), (0, 0, 0)), (8, (2, 4, 2, 2, 2, 2), (0, 0, 0)), (12, (4, 6, 2, 2, 2, 2), (0, 0, 0)),
    (16, (4, 4, 0, 0, 3, 3), (0, 1, 0)), (20, (0, 6, 3, 3, 2, 2), (0, 0, 0)), (22, (5, 5, 2, 2, 2, 2), (0, 0, 0)),
    (64, (0, 0, 0, 0, 2, 2), (1, 1, 0)), (66, (0, 0, 0, 0, 2, 2), (1, 1, 0)), (67, (3, 4, 2, 2, 2, 2), (0, 0, 0)),
    (132, (7, 10, 2, 2, 2, 2), (0, 0, 0)), (260, (10, 10, 3, 3, 2, 2), (0, 0, 0))])
@pytest.mark.parametrize("dtype,n_iso", [("f32", 1), ("f32", 3), ("f64", 1)])
def test_group_updates_give_the_bits_of_the_tile_updates(nx, cpml, periodic, dtype, n_iso):
    sc = _scene(nx, cpml, periodic, n_iso, dtype)
    if n_iso == 3:   # an anisotropic cell inside a slab must pass the admission rule
        for a in sc.inv_eps[1:]:
            a[...] = sc.inv_eps[0]
        sc.inv_eps[2][5, 6, cpml[0]:nx - cpml[1]] = 0.5
    ref = _run(sc, dtype, 0)
    for got in (_run(sc, dtype, 4), _run(sc, dtype, 4, shift=2), _run(sc, dtype, 4, shift=1)):
        for a, b in zip(ref, got):
            assert torch.equal(a, b)


@pytest.mark.parametrize("nx,n_poles", [(24, 1), (24, 2), (26, 2), (27, 2), (32, 3), (33, 5)])
def test_group_pole_updates_give_the_bits_of_the_tile_updates(nx, n_poles):
    sc = _scene(nx, (3, 3, 2, 2, 2, 2), (0, 0, 0), 1, "f32", poles=n_poles)
    ref, got = _run(sc, "f32", 0), _run(sc, "f32", 4)
    for a, b in zip(ref, got):
        assert torch.equal(a, b)


def _transposed(sc, dtype, mode, design):
    """The adjoint state and the material cotangent after six transposed steps from a random adjoint state."""
    ctx = fdtd.Context(sc, dtype=dtype)
    fdtd.fdtd_set_launch_mode(ctx.ctx, mode)
    nx, ny, nz = sc.shape
    ctx.step(6)
    grad = None
    if design is not None:
        lo, hi = design
        grad = torch.zeros(3 * int(np.prod([h - l for l, h in zip(lo, hi)])), dtype=torch.float64, device="cuda")
        fdtd.fdtd_set_design(ctx.ctx, 0, lo, hi, grad.data_ptr())
    fdtd.fdtd_adjoint_begin(ctx.ctx)
    rng = np.random.default_rng(nx)
    for p in range(18):
        n = fdtd.fdtd_part_size(ctx.ctx, 0, p)
        v = rng.standard_normal(n)
        if p < 3:   # E nodes a wall holds carry nothing
            a = v.reshape(nz, ny, nx)
            for q in range(3):
                if q != p and not sc.periodic[q]:
                    a[(slice(None),) * (2 - q) + (0,)] = 0.0
        ctx.set_part(0, p, torch.from_numpy(v), which=1)
    for m in range(6):
        fdtd.fdtd_set_step_count(ctx.ctx, 5 - m)   # the held forward state stands in for every u^m
        fdtd.fdtd_step_adjoint(ctx.ctx, 1)
    out = [ctx.part(0, p, which=1).double() for p in range(18)] + ([grad] if grad is not None else [])
    ctx.close()
    return out


@pytest.mark.parametrize("nx,cpml,periodic,design", [
    (2, (0, 0, 2, 2, 2, 2), (0, 0, 0), None), (4, (0, 0, 2, 2, 0, 3), (1, 0, 0), None),
    (7, (2, 3, 0, 2, 2, 0), (0, 0, 0), None), (8, (2, 4, 2, 2, 2, 2), (0, 0, 0), None),
    (12, (4, 6, 2, 2, 2, 2), (0, 0, 0), None), (16, (4, 4, 0, 0, 3, 3), (0, 1, 0), ((5, 0, 4), (9, 13, 7))),
    (20, (0, 6, 3, 3, 2, 2), (0, 0, 0), ((0, 4, 3), (14, 5, 8))), (22, (5, 5, 2, 2, 2, 2), (0, 0, 0), None),
    (37, (3, 4, 2, 2, 2, 2), (0, 0, 0), ((17, 3, 4), (20, 9, 5))),
    (66, (0, 0, 0, 0, 2, 2), (1, 1, 0), ((60, 0, 3), (66, 4, 9))), (132, (7, 10, 2, 2, 2, 2), (0, 0, 0), None)])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_transposed_group_updates_agree_with_the_tile_updates(nx, cpml, periodic, design, dtype):
    # the two modes round differently: a step is about 20 operations a value, so six steps differ by less than
    # 6 * 20 * eps = 1.4e-5 (FP32), 2.7e-14 (FP64) of the parts' norms; a memory part may be small beside the
    # fields that feed it, so every part is held to the norm of the whole state
    sc = _scene(nx, cpml, periodic, 1, dtype)
    ref, got = _transposed(sc, dtype, 0, design), _transposed(sc, dtype, 4, design)
    tol = 1.4e-5 if dtype == "f32" else 2.7e-14
    norm = max(float(v.norm()) for v in ref[:18])
    for a, b in zip(ref[:18], got[:18]):
        assert float((a - b).norm()) <= tol * norm
    if design is not None:
        assert float(ref[18].norm()) > 0
        assert float((ref[18] - got[18]).norm()) <= tol * float(ref[18].norm())


@pytest.mark.parametrize("nx,n_iso,domains,dtype", [(8, 1, 1, "f64"), (21, 3, 1, "f64"), (36, 1, 3, "f64"), (36, 3, 2, "f32")])
def test_energy_record_of_the_group_updates_is_that_of_the_tile_updates(nx, n_iso, domains, dtype):
    # FP64 sums of about 10^4 terms in another order: each partial sum rounds by eps / 2 of at most the total, so the
    # records differ by less than 10^4 * 1.1e-16 = 1.1e-12 of it (the fields are the same bits)
    scs = [_scene(nx + 2 * q, (0,) * 6, (0, 0, 0), n_iso, dtype) for q in range(domains)]
    out = []
    for mode in (0, 4):
        ctx = fdtd.Context(scs, dtype=dtype)
        fdtd.fdtd_enable_energy(ctx.ctx, 40)
        fdtd.fdtd_set_launch_mode(ctx.ctx, mode)
        ctx.step(35)
        ctx.step(2)
        out.append([(ctx.energy(d, 37), ctx.part(d, 3).clone()) for d in range(domains)])
        ctx.close()
    for (wa, fa), (wb, fb) in zip(*out):
        assert torch.equal(fa, fb)
        assert wa[-1] > 0
        assert np.all(np.abs(wa - wb) <= 1.1e-12 * np.abs(wa).max())
