"""One launch steps every domain of a batch, whatever their number: the bits of the tile launches."""
import pytest

torch = pytest.importorskip("torch")

from paper_2609_30039_gb300 import fdtd as F  # noqa: E402
from paper_2609_30039_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _scene(nx, ny, nz):
    c = (nx // 2, ny // 2, nz // 2)
    return W.Scene(shape=(nx, ny, nz), n_steps=20, sources=[W.Source(W.EZ, c, tuple(v + 1 for v in c),
                                                                    W.gaussian_pulse(20, 8.0, periods=0.3, delay=1.0))])


def _forward(scenes, mode):
    ctx = F.Context(scenes, dtype="f32")
    F.fdtd_set_launch_mode(ctx.ctx, mode)
    ctx.step(9)
    out = [ctx.part(d, p).clone() for d in range(len(scenes)) for p in range(ctx.part_count(d))]
    ctx.close()
    return out


@pytest.mark.parametrize("count", [2, 31, 32, 33, 64, 65, 1025])
def test_every_domain_of_a_batch_is_stepped(count):
    # uneven domains (so uneven numbers of blocks), a point source in each
    scs = [_scene(4 + 2 * (d % 4), 4 + d % 3, 4 + d % 5) for d in range(count)]
    a, b = _forward(scs, 0), _forward(scs, 4)
    assert len(a) == len(b)
    assert all(float(x.abs().sum()) > 0 for x in b[2::18])   # Ez of every domain
    for x, y in zip(a, b):
        assert torch.equal(x, y)
