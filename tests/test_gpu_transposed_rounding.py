"""A transposed step in FP32 rounds no product of the Courant number by itself: it has the bits of the sums with every
product fused into the addition that takes it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2609_30039_gb300 import fdtd as F  # noqa: E402
from paper_2609_30039_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

F32 = np.float32


def _fma(a, b, c):
    """a b + c rounded once to FP32 (the FP64 product of FP32 values is exact; its sum rounds 29 bits further down)."""
    return (np.float64(a) * np.float64(b) + np.float64(c)).astype(F32)


def _back(a, axis):
    """a at the -1 neighbour along a (z, y, x) axis, zero beyond the wall."""
    out = np.zeros_like(a)
    src = [slice(None)] * 3
    dst = [slice(None)] * 3
    src[axis], dst[axis] = slice(0, -1), slice(1, None)
    out[tuple(dst)] = a[tuple(src)]
    return out


def _held(c, shape):
    """Nodes of E_c that the walls at coordinate 0 hold."""
    m = np.zeros(shape, dtype=bool)
    for q in range(3):
        if q != c:
            m[(slice(None),) * (2 - q) + (0,)] = True
    return m


def _step(sc, parts):
    """The adjoint parts after one transposed step from the given ones."""
    ctx = F.Context(sc, dtype="f32")
    F.fdtd_set_step_count(ctx.ctx, 2)
    F.fdtd_adjoint_begin(ctx.ctx)
    for p, v in parts.items():
        ctx.set_part(0, p, torch.from_numpy(v.reshape(-1)), which=1)
    F.fdtd_step_adjoint(ctx.ctx, 1)
    out = {p: ctx.part(0, p, which=1).cpu().numpy().reshape(v.shape) for p, v in parts.items()}
    ctx.close()
    return out


def _fields(rng, shape):
    f = {c: rng.standard_normal(shape).astype(F32) for c in range(6)}
    for c in range(3):
        f[c][_held(c, shape)] = 0
    return f


@pytest.mark.parametrize("nx,ny,nz", [(40, 36, 32), (38, 35, 33), (37, 35, 33)])
def test_gathered_terms_are_fused(nx, ny, nz):
    # S eps^-1 is one, so the lagged form and its completion leave Ebar as the step makes it
    S = F32(W.COURANT)
    inv = F32(1.0) / S
    assert S * inv == 1
    f = _fields(np.random.default_rng(nx), (nz, ny, nx))
    got = _step(W.Scene(shape=(nx, ny, nz), n_steps=8, inv_eps=[np.full((nz, ny, nx), np.float64(inv))]), f)
    for c in range(3):
        c1, c2 = (c + 1) % 3, (c + 2) % 3
        h1, h2 = f[3 + c1], f[3 + c2]
        # the derivatives along c2 of H_c1 and along c1 of H_c2, both with the -1 neighbour ((z, y, x) arrays)
        want = _fma(S, (h1 - _back(h1, 2 - c2)) - (h2 - _back(h2, 2 - c1)), f[c])
        keep = ~_held(c, (nz, ny, nx))
        assert np.array_equal(got[c][keep], want[keep]), c


@pytest.mark.parametrize("nx", [24, 22, 21])
def test_memories_of_h_are_fused(nx):
    ny, nz, d = 20, 18, 4
    S = F32(W.COURANT)
    sc = W.Scene(shape=(nx, ny, nz), n_steps=8, cpml=(0, 0, 0, 0, d, d), kappa_max=3.0, alpha_max=0.05)
    rng = np.random.default_rng(nx)
    f = _fields(rng, (nz, ny, nx))
    mem = {p: rng.standard_normal((2 * d, ny, nx)).astype(F32) for p in (13, 14)}   # of H_x and H_y, along z
    got = _step(sc, {**f, **mem})
    planes = np.r_[0:d, nz - d:nz]
    x = planes + 0.5   # depth of the half-integer node in its slab
    rho = np.where(planes < d, d - x, x - (nz - d)) / d
    sigma, kappa, alpha = 0.8 * 4.0 * rho ** 3, 1.0 + 2.0 * rho ** 3, 0.05 * (1.0 - rho)
    b = np.exp(-(sigma / kappa + alpha) * W.COURANT).astype(F32)[:, None, None]
    assert np.array_equal(got[13], b * _fma(S, f[3][planes], mem[13]))
    assert np.array_equal(got[14], b * _fma(-S, f[4][planes], mem[14]))
