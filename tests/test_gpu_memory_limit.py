"""Snapshots when device memory runs out: the library's objects are linked once more with cudaMalloc and cudaFree behind a
byte limit (the failure is the host's: nothing is allocated beyond it), and a save that fails leaves the slots as they were."""
import os
import subprocess
import sys
import textwrap

import pytest

torch = pytest.importorskip("torch")

from paper_2609_30039_gb300 import build as B  # noqa: E402

pytestmark = pytest.mark.gpu

WRAP = r"""
#include <cstddef>
#include <map>
extern "C" {
int __real_cudaMalloc(void** p, size_t bytes);
int __real_cudaFree(void* p);
static long long left = -1;
static std::map<void*, size_t>* sizes = nullptr;
void limit_bytes(long long n) { left = n; }   // -1: no limit
int __wrap_cudaMalloc(void** p, size_t bytes) {
    if (!sizes) sizes = new std::map<void*, size_t>;
    if (left >= 0 && (long long)bytes > left) return 2;   // cudaErrorMemoryAllocation
    const int e = __real_cudaMalloc(p, bytes);
    if (e == 0) {
        (*sizes)[*p] = bytes;
        if (left >= 0) left -= (long long)bytes;
    }
    return e;
}
int __wrap_cudaFree(void* p) {
    if (sizes && p && sizes->count(p)) {
        if (left >= 0) left += (long long)(*sizes)[p];
        sizes->erase(p);
    }
    return __real_cudaFree(p);
}
}
"""

HEAD = """
import sys
sys.path.insert(0, {root!r})
import ctypes as C
import torch
from paper_2609_30039_gb300 import fdtd as F
lib = F.load({lib!r})
lib.limit_bytes.argtypes = [C.c_longlong]
from tests.test_gpu_schedule_errors import _Run, _halves, _same, _scene

def parts(ctx):
    return [ctx.part(0, p).clone() for p in range(ctx.part_count(0))]

def equal(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))
"""


@pytest.fixture(scope="module")
def limited(tmp_path_factory):
    """Runs a script against the library with the limit."""
    d = tmp_path_factory.mktemp("limited")
    src, obj, lib = str(d / "limit.cpp"), str(d / "limit.o"), str(d / "libgbfdtd.so")
    with open(src, "w") as f:
        f.write(WRAP)
    subprocess.run(["g++", "-O1", "-fPIC", "-c", src, "-o", obj], check=True)
    objs = [os.path.join(B.OBJ_DIR, os.path.basename(s)[:-3] + ".o") for s in B.sources()]
    if not all(os.path.exists(o) for o in objs):   # a library built elsewhere, without its objects
        B.build(force=True)
    subprocess.run([B._nvcc(), *B.ARCH, "-shared", "-o", lib, obj, *objs, "-Xlinker", "--wrap=cudaMalloc", "-Xlinker",
                    "--wrap=cudaFree"], check=True)

    def run(body):
        code = HEAD.format(root=B.ROOT, lib=lib) + textwrap.dedent(body)
        r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300, cwd=B.ROOT)
        assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]

    return run


def test_a_save_without_memory_leaves_the_slot(limited):
    limited("""
        ctx = F.Context([_scene()], dtype="f32")
        c = ctx.ctx
        ctx.step(5)
        want = parts(ctx)
        F.fdtd_state_save(c, 0, F.FDTD_CODEC_NATIVE)
        ctx.step(3)
        lib.limit_bytes(0)   # the table of the other codec does not fit
        assert lib.fdtd_state_save(c, 0, F.FDTD_CODEC_BF16) == F.FDTD_ENOMEM
        lib.limit_bytes(-1)
        F.fdtd_state_restore(c, 0)
        assert ctx.step_count == 5 and equal(want, parts(ctx))
        ctx.close()
        """)


@pytest.mark.parametrize("codec", ["FDTD_CODEC_NATIVE", "FDTD_CODEC_BF16"])
def test_a_first_save_without_memory_leaves_the_slot_empty(limited, codec):
    limited(f"""
        ctx = F.Context([_scene()], dtype="f32")
        c = ctx.ctx
        ctx.step(5)
        size = F.fdtd_snapshot_bytes(c, F.{codec})
        for room in (0, size - 1):   # nothing, the table alone
            lib.limit_bytes(room)
            assert lib.fdtd_state_save(c, 0, F.{codec}) == F.FDTD_ENOMEM
            lib.limit_bytes(-1)
            assert lib.fdtd_state_restore(c, 0) == F.FDTD_ESTATE
        ctx.close()
        ctx = F.Context([_scene()], dtype="f32")
        lib.limit_bytes(size)   # the slot or the table, not both
        assert lib.fdtd_state_save(ctx.ctx, 0, F.{codec}) == F.FDTD_ENOMEM
        lib.limit_bytes(-1)
        assert lib.fdtd_state_restore(ctx.ctx, 0) == F.FDTD_ESTATE
        F.fdtd_state_save(ctx.ctx, 0, F.{codec})
        F.fdtd_state_restore(ctx.ctx, 0)
        ctx.close()
        """)


def test_a_schedule_without_memory_stops_where_the_single_calls_do(limited):
    limited("""
        steps, slots = 9, 4
        first, rows = _halves(steps, slots)
        for room in range(5):   # slots that fit, and 64 KiB for the rest
            out = []
            for native in (True, False):
                r = _Run([_scene()])
                size = F.fdtd_snapshot_bytes(r.ctx.ctx, F.FDTD_CODEC_NATIVE)
                lib.limit_bytes(room * size + 65536)
                got = [r.run(first, native)]
                if got[0][0] == F.FDTD_OK:
                    r.objective()
                    # the reversal saves two slots that the forward half has not
                    got.append(r.run(rows[:6] + [(0, 7)] + rows[6:] + [(0, 8)], native))
                lib.limit_bytes(-1)
                out.append(got + r.outcome([*range(slots), 7, 8]))
                r.close()
            _same(*out)
        """)
