"""A caller may capture a context's eager steps into a CUDA graph of its own and replay it: the library does not see the
state change, so a restore after the replay must load the slot."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2609_30039_gb300 import fdtd as F  # noqa: E402
from paper_2609_30039_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _scene(n=64):
    rng = np.random.default_rng(3)
    nx, ny, nz, d = 20, 18, 16, 3
    inv = np.ones((nz, ny, nx))
    inv[5:11, 5:13, 6:14] = rng.uniform(0.2, 1.0, size=(6, 8, 8))
    return W.Scene(shape=(nx, ny, nz), n_steps=n, cpml=(d,) * 6, kappa_max=3.0, alpha_max=0.05, inv_eps=[inv],
                   sources=[W.Source(W.EX, (4, 4, 4), (16, 14, 5), W.gaussian_pulse(n, 8.0, periods=0.4, delay=1.0))])


def _state(ctx):
    out = [ctx.part(0, p).clone() for p in range(ctx.part_count(0))]
    ctx.synchronize()
    return out


def _captured(ctx, stream, n):
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        g.capture_begin(capture_error_mode="thread_local")
        ctx.step(n)
        g.capture_end()
    return g


@pytest.mark.parametrize("schedule", [False, True])
def test_restore_after_a_replayed_graph_of_steps_loads_the_slot(schedule):
    stream = torch.cuda.Stream()
    ctx = F.Context(_scene(), dtype="f32", stream=stream)
    c = ctx.ctx
    ctx.step(9)
    g = _captured(ctx, stream, 4)
    F.fdtd_set_step_count(c, 9)   # the captured steps have not run
    want = _state(ctx)
    acts = np.array([[F.FDTD_ACT_SAVE, 0]], dtype=np.int32)
    back = np.array([[F.FDTD_ACT_RESTORE, 0]], dtype=np.int32)
    if schedule:
        F.fdtd_run_schedule(c, acts, 0, F.FDTD_CODEC_NATIVE)
    else:
        F.fdtd_state_save(c, 0, F.FDTD_CODEC_NATIVE)
    with torch.cuda.stream(stream):
        g.replay()
    moved = _state(ctx)
    assert any(not torch.equal(a, b) for a, b in zip(want, moved))
    if schedule:
        F.fdtd_run_schedule(c, back, 0, F.FDTD_CODEC_NATIVE)
    else:
        F.fdtd_state_restore(c, 0)
    got = _state(ctx)
    assert ctx.step_count == 9
    for a, b in zip(want, got):
        assert torch.equal(a, b)
    # the replay steps on from the step count of the device: the same four steps as eager ones
    ctx.step(4)
    for a, b in zip(moved, _state(ctx)):
        assert torch.equal(a, b)
    ctx.close()
