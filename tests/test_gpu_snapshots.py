"""The native schedule executor leaves out snapshot copies that nothing needs, and one launch codes a whole BF16
snapshot: both must give the bits of the plain calls and of the codec's definition."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2609_30039_gb300 import adjoint as A  # noqa: E402
from paper_2609_30039_gb300 import fdtd as F  # noqa: E402
from paper_2609_30039_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _scene(nx=20, poles=0, n=32):
    ny, nz, d = 18, 16, 3
    rng = np.random.default_rng(nx)
    inv = np.ones((nz, ny, nx))
    inv[5:11, 5:13, 6:14] = rng.uniform(0.2, 1.0, size=(6, 8, 8))
    mask = np.zeros((nz, ny, nx), dtype=np.uint8)
    mask[6:9, 6:12, 7:13] = 1
    pl = tuple((W.LORENTZ, 1.0 + p, 0.1, 0.01) for p in range(poles))
    return W.Scene(shape=(nx, ny, nz), n_steps=n, cpml=(d,) * 6, kappa_max=3.0, alpha_max=0.05, inv_eps=[inv],
                   poles=pl, pole_mask=mask if poles else None,
                   sources=[W.Source(W.EX, (4, 4, 4), (16, 14, 5), W.gaussian_pulse(n, 8.0, periods=0.4, delay=1.0))],
                   monitors=[W.Monitor((7, 7, 11), (13, 12, 12), (W.EX,), W.omegas_for((8.0, 9.0)))],
                   design=((6, 5, 5), (14, 13, 11)))


def _gradient(poles, steps, slots, codec, native):
    """Gradient, final state and slot contents of a replay; native: the library's executor, else one call per action."""
    sc = _scene(poles=poles)
    ctx = F.Context(sc, dtype="f32")
    g = torch.zeros(3 * 8 * 8 * 6, dtype=torch.float64, device="cuda")
    F.fdtd_set_design(ctx.ctx, 0, sc.design[0], sc.design[1], g.data_ptr())
    acts = A.schedule(steps, slots)
    keep = []

    def objective(cx):
        keep.append((2.0 * cx.dft(0)).contiguous())
        F.fdtd_set_adjoint_source(cx.ctx, cx.monitors[0][0], keep[-1].data_ptr())
        return 0.0

    if native:
        A.run_schedule(ctx, acts, objective, codec)
    else:
        c = ctx.ctx
        for a in acts:
            if a[0] == "save":
                F.fdtd_state_save(c, a[1], codec)
            elif a[0] == "restore":
                F.fdtd_state_restore(c, a[1])
            elif a[0] == "advance":
                F.fdtd_step_forward(c, a[1])
            elif a[0] == "adjoint":
                F.fdtd_step_adjoint(c, 1)
            else:
                objective(ctx)
                F.fdtd_adjoint_begin(c)
                F.fdtd_dft_enable(c, 0)
    ctx.synchronize()
    out = [g.clone(), torch.tensor([ctx.step_count])]
    out += [ctx.part(0, p, which=w).clone() for w in (0, 1) for p in range(ctx.part_count(0))]
    for s in sorted({a[1] for a in acts if a[0] == "save"}):
        F.fdtd_state_restore(ctx.ctx, s)
        out += [torch.tensor([ctx.step_count])] + [ctx.part(0, p).clone() for p in range(ctx.part_count(0))]
    ctx.close()
    return out


@pytest.mark.parametrize("steps,slots", [(1, 1), (2, 1), (5, 1), (6, 2), (13, 3), (24, 4), (24, 24)])
@pytest.mark.parametrize("poles", [0, 2])
@pytest.mark.parametrize("codec", [F.FDTD_CODEC_NATIVE, F.FDTD_CODEC_BF16])
def test_native_schedule_gives_the_bits_of_single_calls(steps, slots, poles, codec):
    a, b = (_gradient(poles, steps, slots, codec, native) for native in (True, False))
    # (a signal moves at most one plane a step: the monitor, 7 planes on, sees nothing of the shortest runs)
    assert float(a[0].abs().sum()) > 0 or steps <= 7
    assert len(a) == len(b)
    # pole states go through one FP64 gradient per cell and step either way: every output is the same
    for x, y in zip(a, b):
        assert torch.equal(x, y)


@pytest.mark.parametrize("nx", [20, 21, 22])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_bf16_snapshot_is_one_scale_per_slab(nx, dtype):
    sc = _scene(nx=nx, poles=2)
    ctx = F.Context(sc, dtype=dtype)
    rng = np.random.default_rng(nx)
    parts = []
    for p in range(ctx.part_count(0)):
        n = F.fdtd_part_size(ctx.ctx, 0, p)
        v = rng.standard_normal(n) * 10.0 ** rng.integers(-30, 30)
        if p == 2:
            v[: n // 2] = 0.0          # zero slabs
        if p == 4:
            v[:] = 1e-42               # an FP32 denormal maximum
        parts.append(torch.from_numpy(v).to(ctx.tdtype).cuda())
        ctx.set_part(0, p, parts[-1])
    F.fdtd_state_save(ctx.ctx, 3, F.FDTD_CODEC_BF16)
    ctx.step(3)
    F.fdtd_state_restore(ctx.ctx, 3)
    lo, hi = F.fdtd_ade_box(ctx.ctx, 0)
    for p, v in enumerate(parts):
        if p < 6:
            planes = 16
        elif p < 18:
            a, s = ((p - 6) % 6) // 2, (p - 6) % 2
            planes = 6 if (a + 1 + s) % 3 == 2 else 16
        else:
            planes = hi[2] - lo[2]
        x = v.float().view(planes, -1)
        s = x.abs().amax(1, keepdim=True)
        q = torch.where(s > 0, x / torch.where(s > 0, s, torch.ones_like(s)), torch.zeros_like(x)).bfloat16().float()
        assert torch.equal(ctx.part(0, p), (q * s).reshape(-1).to(ctx.tdtype)), p
    ctx.close()


def test_snapshot_of_a_state_changed_since_is_restored():
    # each way the state can change between a save and a restore of the same slot
    sc = _scene()
    ctx = F.Context(sc, dtype="f32")
    ctx.step(9)
    F.fdtd_state_save(ctx.ctx, 0, F.FDTD_CODEC_NATIVE)
    want = [ctx.part(0, p).clone() for p in range(18)]

    def step():
        ctx.step(1)

    def part():
        ctx.set_part(0, 3, torch.zeros_like(want[3]))

    def reset():
        F.fdtd_reset(ctx.ctx)

    def time():
        F.fdtd_time_half_steps(ctx.ctx, 0, 2)

    def tune():
        F.fdtd_autotune(ctx.ctx, 4)

    def other():
        ctx.step(2)
        F.fdtd_state_save(ctx.ctx, 1, F.FDTD_CODEC_NATIVE)

    def lossy():
        F.fdtd_state_save(ctx.ctx, 1, F.FDTD_CODEC_BF16)
        F.fdtd_state_restore(ctx.ctx, 1)

    for change in (step, part, reset, time, tune, other, lossy, lambda: F.fdtd_set_step_count(ctx.ctx, 77)):
        change()
        F.fdtd_state_restore(ctx.ctx, 0)
        assert ctx.step_count == 9
        for p in range(18):
            assert torch.equal(ctx.part(0, p), want[p])
    F.fdtd_snapshots_free(ctx.ctx)
    with pytest.raises(F.FdtdError):
        F.fdtd_state_restore(ctx.ctx, 0)
    ctx.close()
