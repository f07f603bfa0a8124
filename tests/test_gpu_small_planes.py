"""Planes that fit one block of threads take shorter groups and one region: the bits of the tile launches (transposed: of
one cell per thread) all the same."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2609_30039_gb300 import fdtd as F  # noqa: E402
from paper_2609_30039_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _scene(nx, ny, nz, cpml, periodic=(0, 0, 0), poles=0, n_iso=1, monitor=True):
    n = 20
    rng = np.random.default_rng(100 * nx + ny)
    inv = [np.ones((nz, ny, nx)) for _ in range(n_iso)]
    mid = (slice(cpml[4], nz - cpml[5]), slice(cpml[2], ny - cpml[3]), slice(cpml[0], nx - cpml[1]))
    for a in inv:
        a[mid] = rng.uniform(0.2, 1.0, size=a[mid].shape)
    c = (nx // 2, ny // 2, nz // 2)
    src = [W.Source(W.EZ, c, tuple(v + 1 for v in c), W.gaussian_pulse(n, 8.0, periods=0.3, delay=1.0))]
    mons = [W.Monitor((0, 0, 3), (nx, ny, 5), (W.EX, W.HZ), W.omegas_for((8.0, 9.0)))] if monitor else []
    mask = None
    if poles:
        mask = np.zeros((nz, ny, nx), dtype=np.uint8)
        mask[3:nz - 3, cpml[2]:ny - cpml[3], cpml[0] + 1:nx - cpml[1]] = 1
    pl = tuple((W.LORENTZ, 1.0 + p, 0.1 + 0.05 * p, 0.01) for p in range(poles))
    return W.Scene(shape=(nx, ny, nz), n_steps=n, cpml=cpml, kappa_max=3.0, alpha_max=0.05, inv_eps=inv, sources=src,
                   monitors=mons, periodic=periodic, poles=pl, pole_mask=mask)


def _forward(scenes, dtype, mode):
    ctx = F.Context(scenes, dtype=dtype)
    F.fdtd_set_launch_mode(ctx.ctx, mode)
    ctx.step(9)
    out = [ctx.part(d, p).clone() for d in range(len(scenes)) for p in range(ctx.part_count(d))]
    out += [ctx.dft(k).clone() for k in range(len(ctx.monitors))]
    ctx.close()
    return out


PLANES = [(2, 2), (4, 8), (8, 8), (8, 16), (12, 12), (16, 16), (4, 64), (2, 64), (16, 17), (6, 10), (10, 26), (20, 20), (32, 16)]


@pytest.mark.parametrize("nx,ny", PLANES)
@pytest.mark.parametrize("kind", ["slabs", "periodic", "poles", "aniso"])
def test_small_planes_give_the_bits_of_the_tile_updates(nx, ny, kind):
    x = (1, 1) if nx >= 4 else (0, 0)
    y = (2, 1) if ny >= 8 else (0, 0)
    sc = {"slabs": lambda: _scene(nx, ny, 11, x + y + (2, 2)),
          "periodic": lambda: _scene(nx, ny, 11, (0, 0, 0, 0, 2, 2), periodic=(1, 1, 0)),
          "poles": lambda: _scene(nx, ny, 11, x + y + (2, 2), poles=2),
          "aniso": lambda: _scene(nx, ny, 11, (0,) * 6, n_iso=3)}[kind]()
    for dtype in ("f32", "f64"):
        for a, b in zip(_forward([sc], dtype, 0), _forward([sc], dtype, 4)):
            assert torch.equal(a, b)


def _transposed(sc, shift):
    """The adjoint state after five transposed steps from a random one; shift: eps^-1 off its 16-byte boundary, so that every
    thread takes one cell."""
    ctx = F.Context(sc, dtype="f32")
    nx, ny, nz = sc.shape
    if shift:
        buf = torch.empty(nx * ny * nz + 1, dtype=torch.float32, device="cuda")
        buf[1:] = ctx.inv_eps[0][0].reshape(-1)
        ctx.set_inv_eps(0, [buf[1:].view(nz, ny, nx)] * 3)
    ctx.step(6)
    F.fdtd_adjoint_begin(ctx.ctx)
    rng = np.random.default_rng(nx)
    for p in range(18):
        v = rng.standard_normal(F.fdtd_part_size(ctx.ctx, 0, p))
        if p < 3:   # E nodes a wall holds carry nothing
            a = v.reshape(nz, ny, nx)
            for q in range(3):
                if q != p and not sc.periodic[q]:
                    a[(slice(None),) * (2 - q) + (0,)] = 0.0
        ctx.set_part(0, p, torch.from_numpy(v), which=1)
    F.fdtd_step_adjoint(ctx.ctx, 5)
    out = [ctx.part(0, p, which=1).clone() for p in range(18)]
    ctx.close()
    return out


@pytest.mark.parametrize("nx,ny,nz", [(*p, 11) for p in PLANES] + [(8, 8, 1300), (12, 12, 1217), (16, 16, 1216)])
@pytest.mark.parametrize("kind", ["slabs", "periodic"])
def test_small_planes_transposed_give_the_bits_of_single_cells(nx, ny, nz, kind):
    x = (1, 1) if nx >= 4 else (0, 0)
    y = (2, 1) if ny >= 8 else (0, 0)
    sc = _scene(nx, ny, nz, x + y + (2, 2), monitor=False) if kind == "slabs" else \
        _scene(nx, ny, nz, (0, 0, 0, 0, 2, 2), periodic=(1, 1, 0), monitor=False)
    for a, b in zip(_transposed(sc, True), _transposed(sc, False)):
        assert torch.equal(a, b)
