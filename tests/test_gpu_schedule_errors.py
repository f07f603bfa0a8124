"""The native schedule executor leaves out copies; its outcome is that of one call per action all the same: where an action
fails, over several domains, in both launch modes, and where a run ends."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2609_30039_gb300 import adjoint as A  # noqa: E402
from paper_2609_30039_gb300 import fdtd as F  # noqa: E402
from paper_2609_30039_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

SAVE, RESTORE, ADVANCE, ADJOINT, STOP = range(5)
MISSING = 99


def _scene(nx=20, ny=18, nz=16, design=((6, 5, 5), (14, 13, 11)), periodic=(0, 0, 0), zlo=3, n=32):
    d = 3
    rng = np.random.default_rng(nx + nz)
    inv = np.ones((nz, ny, nx))
    inv[5:9, 5:9, 6:12] = rng.uniform(0.2, 1.0, size=(4, 4, 6))
    cp = (0, 0) if periodic[0] else (d, d)
    return W.Scene(shape=(nx, ny, nz), n_steps=n, cpml=cp + (d, d, zlo, d), kappa_max=3.0, alpha_max=0.05, inv_eps=[inv],
                   periodic=periodic,
                   sources=[W.Source(W.EX, (4, 4, 4), (nx - 4, ny - 4, 5), W.gaussian_pulse(n, 8.0, periods=0.4, delay=1.0))],
                   monitors=[W.Monitor((7, 7, 8), (11, 11, 9), (W.EX, W.HY), W.omegas_for((8.0, 9.0)))], design=design)


class _Run:
    """A context with design boxes, stepped by runs of (kind, arg) rows: native, or one call per action."""

    def __init__(self, scenes, mode=4):
        self.ctx = F.Context(scenes, dtype="f32")
        F.fdtd_set_launch_mode(self.ctx.ctx, mode)
        self.grads, self.cots = [], []
        for d, sc in enumerate(scenes):
            if sc.design is None:
                continue
            lo, hi = sc.design
            n = 3 * int(np.prod([h - l for l, h in zip(lo, hi)]))
            self.grads.append(torch.zeros(n, dtype=torch.float64, device="cuda"))
            F.fdtd_set_design(self.ctx.ctx, d, lo, hi, self.grads[-1].data_ptr())

    def objective(self):
        for k in range(len(self.ctx.monitors)):
            self.cots.append((2.0 * self.ctx.dft(k)).contiguous())
            F.fdtd_set_adjoint_source(self.ctx.ctx, self.ctx.monitors[k][0], self.cots[-1].data_ptr())
        F.fdtd_adjoint_begin(self.ctx.ctx)
        F.fdtd_dft_enable(self.ctx.ctx, 0)

    def run(self, rows, native, codec=F.FDTD_CODEC_NATIVE):
        """(status, executed) of one run."""
        lib, c = F.load(), self.ctx.ctx
        if native:
            a = np.ascontiguousarray(rows, dtype=np.int32)
            done = C.c_int32(0)
            st = lib.fdtd_run_schedule(c, a.ctypes.data_as(C.POINTER(C.c_int32)), len(rows), codec, C.byref(done))
            return int(st), int(done.value)
        for i, (kind, arg) in enumerate(rows):
            if kind == STOP:
                return F.FDTD_OK, i + 1
            call = {SAVE: lambda: lib.fdtd_state_save(c, arg, codec), RESTORE: lambda: lib.fdtd_state_restore(c, arg),
                    ADVANCE: lambda: lib.fdtd_step_forward(c, arg), ADJOINT: lambda: lib.fdtd_step_adjoint(c, arg)}.get(kind)
            st = call() if call else F.FDTD_EINVAL
            if st != F.FDTD_OK:
                return int(st), i
        return F.FDTD_OK, len(rows)

    def outcome(self, slots):
        """Step counts, states, gradients, then every slot's status and state."""
        ctx = self.ctx

        def parts(whichs):
            return [ctx.part(d, p, which=w).clone() for d in range(len(ctx.scenes)) for w in whichs
                    for p in range(ctx.part_count(d))]

        out = [ctx.step_count, F.fdtd_adjoint_step_count(ctx.ctx)] + [g.clone() for g in self.grads]
        out += [v.clone() for v in parts((0,))]
        # the device's step count shows in what the sources add
        ctx.step(2)
        out += parts((0, 1))
        for s in slots:
            st = int(F.load().fdtd_state_restore(ctx.ctx, s))
            out.append(st)
            if st == F.FDTD_OK:
                out += [ctx.step_count] + parts((0,))
        ctx.synchronize()
        return out

    def close(self):
        self.ctx.close()


def _same(a, b):
    assert len(a) == len(b)
    for q, (x, y) in enumerate(zip(a, b)):
        assert torch.equal(x, y) if torch.is_tensor(x) else x == y, q


def _halves(steps, slots):
    rows = [tuple(int(v) for v in r) for r in A.encode(A.schedule(steps, slots))]
    cut = [k for k, _ in rows].index(STOP) + 1
    return rows[:cut], rows[cut:]


def _both(scenes, steps, slots, reversal, mode=4, splits=()):
    """Outcome of the forward half and of `reversal`, native and by single calls; splits: where further runs begin."""
    out = []
    first, _ = _halves(steps, slots)
    for native in (True, False):
        r = _Run(scenes, mode)
        got = [r.run(first, native)]
        r.objective()
        edges = [0, *splits, len(reversal)]
        for a, b in zip(edges, edges[1:]):
            got.append(r.run(reversal[a:b], native))
            if got[-1][0] != F.FDTD_OK:
                break
        out.append(got + r.outcome(range(slots)))
        r.close()
    return out


def test_a_failing_action_leaves_what_the_single_calls_leave():
    steps, slots = 9, 3
    _, rows = _halves(steps, slots)
    for at in range(len(rows) + 1):
        for bad in ((RESTORE, MISSING), (ADVANCE, -1), (ADJOINT, steps + 1), (SAVE, -1), (7, 0)):
            a, b = _both([_scene()], steps, slots, rows[:at] + [bad] + rows[at:])
            assert a[1] != (F.FDTD_OK, len(rows) + 1)
            _same(a, b)


def test_steps_in_place_before_a_missing_slot():
    # both slots are saved again after the failing action, and transposed steps alone read them before it
    rows = [(RESTORE, 0), (ADVANCE, 1), (SAVE, 1), (ADVANCE, 1), (SAVE, 2), (RESTORE, 0), (RESTORE, 2), (ADJOINT, 1),
            (RESTORE, 1), (ADJOINT, 1), (RESTORE, MISSING), (SAVE, 1), (SAVE, 2)]
    out = []
    for native in (True, False):
        r = _Run([_scene()])
        got = [r.run([(SAVE, 0), (ADVANCE, 3), (STOP, 0)], native)]
        r.objective()
        got.append(r.run(rows, native))
        out.append(got + r.outcome(range(3)))
        r.close()
    assert out[1][1] == (F.FDTD_ESTATE, 10)
    _same(*out)


@pytest.mark.parametrize("mode", [0, 4])
@pytest.mark.parametrize("name", ["two", "five", "wall", "seam"])
def test_replays_of_several_domains_and_boxes(name, mode):
    if name == "two":   # the second domain has no design box
        scenes = [_scene(), _scene(23, 17, 19, design=None)]
    elif name == "five":
        scenes = [_scene(18 + q, 16, 15 + q, design=((6, 5, 5), (9, 9, 8 + q))) for q in range(5)]
    elif name == "wall":   # against the wall z = 0
        scenes = [_scene(design=((4, 4, 0), (11, 9, 3)), zlo=0)]
    else:                  # against the seam of a periodic axis
        scenes = [_scene(design=((0, 5, 4), (3, 9, 9)), periodic=(1, 0, 0)), _scene(21, design=((18, 5, 4), (21, 9, 9)),
                                                                                  periodic=(1, 0, 0))]
    steps, slots = 13, 4
    _, rows = _halves(steps, slots)
    a, b = _both(scenes, steps, slots, rows, mode)
    assert a[1] == (F.FDTD_OK, len(rows))
    _same(a, b)


@pytest.mark.parametrize("splits", [(1,), (2, 3), (4, 9, 10, 15), tuple(range(1, 20))])
def test_runs_split_anywhere(splits):
    steps, slots = 10, 3
    _, rows = _halves(steps, slots)
    a, b = _both([_scene()], steps, slots, rows, splits=tuple(s for s in splits if s < len(rows)))
    _same(a, b)


def test_a_slot_of_the_other_codec_is_read_before_it_is_saved_over():
    out = []
    for native in (True, False):
        r = _Run([_scene()])
        got = [r.run([(ADVANCE, 4), (SAVE, 0), (ADVANCE, 2), (STOP, 0)], native, F.FDTD_CODEC_BF16)]
        got.append(r.run([(SAVE, 1), (ADVANCE, 1), (RESTORE, 0), (ADVANCE, 1), (SAVE, 0), (SAVE, 1), (RESTORE, 1), (RESTORE, 0)],
                         native))
        out.append(got + r.outcome(range(2)))
        r.close()
    _same(*out)
