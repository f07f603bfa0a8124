"""A medium given by eps^-1 pointers (a, a, b) is the one given by (a, copy of a, b): the same bits, in the boxes of poles
and design cells as outside them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2609_30039_gb300 import fdtd as F  # noqa: E402
from paper_2609_30039_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _scene(poles):
    nx, ny, nz, d, n = 22, 18, 16, 3, 16
    rng = np.random.default_rng(5)
    inv = [np.ones((nz, ny, nx)) for _ in range(3)]
    box = (slice(4, 12), slice(4, 14), slice(4, 18))
    inv[0][box] = inv[1][box] = rng.uniform(0.2, 1.0, size=inv[0][box].shape)
    inv[2][box] = rng.uniform(0.2, 1.0, size=inv[0][box].shape)
    mask = np.zeros((nz, ny, nx), dtype=np.uint8)
    mask[6:9, 6:12, 7:13] = 1
    pl = tuple((W.LORENTZ, 1.0 + p, 0.1, 0.01) for p in range(poles))
    return W.Scene(shape=(nx, ny, nz), n_steps=n, cpml=(d,) * 6, kappa_max=3.0, alpha_max=0.05, inv_eps=inv, poles=pl,
                   pole_mask=mask if poles else None,
                   sources=[W.Source(W.EZ, (4, 4, 4), (16, 14, 5), W.gaussian_pulse(n, 8.0, periods=0.4, delay=1.0))],
                   design=((6, 5, 5), (14, 13, 11)))


def _outputs(sc, dtype, mode, pointers):
    ctx = F.Context(sc, dtype=dtype)
    F.fdtd_set_launch_mode(ctx.ctx, mode)
    t, tz = ctx.inv_eps[0][0], ctx.inv_eps[0][2]
    ctx.set_inv_eps(0, [t, t, tz] if pointers == "aab" else [t, t.clone(), tz])
    grad = torch.zeros(3 * 8 * 8 * 6, dtype=torch.float64, device="cuda")
    F.fdtd_set_design(ctx.ctx, 0, sc.design[0], sc.design[1], grad.data_ptr())
    if sc.poles:
        F.fdtd_set_pole_grad(ctx.ctx, 0, 1)
    ctx.step(12)
    F.fdtd_adjoint_begin(ctx.ctx)
    rng = np.random.default_rng(9)
    for p in range(6):   # a random cotangent of the fields away from the walls' held nodes
        v = np.zeros((16, 18, 22))
        v[3:13, 3:15, 3:19] = rng.standard_normal((10, 12, 16))
        ctx.set_part(0, p, torch.from_numpy(v.reshape(-1)), which=1)
    for m in range(4):
        F.fdtd_set_step_count(ctx.ctx, 11 - m)   # the held forward state stands in for every u^m
        F.fdtd_step_adjoint(ctx.ctx, 1)
    out = [ctx.part(0, p, which=w).clone() for w in (0, 1) for p in range(ctx.part_count(0))] + [grad]
    if sc.poles:
        out.append(torch.from_numpy(F.fdtd_pole_grad(ctx.ctx, 0, len(sc.poles))))
    ctx.synchronize()
    ctx.close()
    return out


@pytest.mark.parametrize("poles", [0, 1, 2])
@pytest.mark.parametrize("dtype,mode", [("f32", 4), ("f64", 4), ("f32", 0)])
def test_uniaxial_pointers_give_the_bits_of_three_arrays(poles, dtype, mode):
    a, b = (_outputs(_scene(poles), dtype, mode, p) for p in ("aab", "abc"))
    assert float(b[-1].abs().sum()) > 0
    for q, (x, y) in enumerate(zip(a[:len(a) - (1 if poles else 0)], b)):
        assert torch.equal(x, y), q
    if poles:
        # the coefficient cotangents are summed by FP64 atomics over at most 6 * 8 * 8 * 3 * 4 terms each, in any order, so
        # they differ by 5e3 * 1.1e-16 of their terms' sizes; the terms may exceed the combined result, up to 1e3 times here
        scale = float(b[-1].abs().max())
        assert float((a[-1] - b[-1]).abs().max()) <= 5e3 * 1.1e-16 * 1e3 * scale
