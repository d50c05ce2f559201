"""What asl_run_layer orders behind what, checked on the CPU: the entry points compiled against a runtime that only logs
launches, event records and waits (fake_cuda_runtime.cpp)."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

from paper_2601_07667_b200 import binding as B
from paper_2601_07667_b200 import build

MAIN, SIDE, SIDE2 = 101, 102, 103                     # streams of device 1
CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or build._nvcc()))), "include")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "libasl_fake.so")
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-Wl,-Bsymbolic", "-I", CUDA_INCLUDE, "-I", build.INCLUDE, "-I", build.CSRC,
                    "-x", "c++", os.path.join(build.CSRC, "asl_api.cu"), os.path.join(here, "fake_cuda_runtime.cpp"), "-o", so],
                   check=True)
    fake = C.CDLL(so)
    fake.fake_log.restype = C.c_char_p
    for name in ("asl_run_layer", "asl_run_join", "asl_run_reset", "asl_plan", "asl_create", "asl_destroy"):
        getattr(fake, name).argtypes = getattr(B.library(), name).argtypes
    fake.fake_fail(b"", 0)
    return fake


class Layers:
    """A context on device 1 with a plan, made and used while device 0 is current."""

    def __init__(self, lib):
        self.lib, self.ctx = lib, C.c_void_p()
        assert lib.asl_create(C.byref(self.ctx), 1) == B.ASL_OK
        cu, bu = (C.c_int32 * 2)(0, 1000), (C.c_int32 * 1)(100)
        p = B.AslParams(8, 2, 128, 32, 7, 0, 1, 1, 2, 0, 0.3, cu, bu, (C.c_int64 * 3)(8 * 32 * 128, 32 * 128, 128),
                        (C.c_int64 * 2)(256, 128), (C.c_int64 * 2)(256, 128), 0, 0, None)
        size = C.c_size_t()
        assert lib.asl_plan(self.ctx, C.byref(p), C.byref(size)) == B.ASL_OK
        self.size = size.value
        lib.fake_clear()

    def run(self, slot, one_side=0, n_rows=1, idx=0x1000):
        a = 0x1000                                     # never looked at
        layer = B.AslLayer(a, self.size, (C.c_void_p * 2)(a, a), (C.c_void_p * 2)(a, a), a, a, idx, a, a, MAIN, SIDE, SIDE2, one_side, 0)
        return self.lib.asl_run_layer(self.ctx, C.byref(layer), a, a, a, None, 1, n_rows, slot)

    def order(self):
        """(name of every launch so far, what lies before it, what each stream has behind it)."""
        names, before, streams, events = [], [], {}, {}
        for line in self.lib.fake_log().decode().splitlines():
            what, a, b = line.split()
            st = int(b)
            if what == "run":
                before.append(frozenset(streams.get(st, frozenset())))
                streams[st] = streams.get(st, frozenset()) | {len(names)}
                names.append(a)
            elif what == "record":
                events[a] = streams.get(st, frozenset())
            else:
                streams[st] = streams.get(st, frozenset()) | events[a]
        return names, before, streams

    def close(self):
        assert self.lib.asl_destroy(self.ctx) == B.ASL_OK


@pytest.mark.parametrize("one_side", [0, 1])
@pytest.mark.parametrize("fail,issued", [
    ("pool", ["score"]), ("rank", ["score", "pool"]), ("topk", ["score", "pool", "rank"]),
    ("compact", ["score", "pool", "rank", "topk"]),
    (dict(n_rows=3), ["score", "pool"]), (dict(idx=None), ["score", "pool", "rank"]),      # refused by a step's own checks
])
def test_a_slot_waits_for_what_a_failed_layer_left_in_flight(lib, fail, issued, one_side):
    """A step of a layer fails when the steps before it are already queued: the slot's next scoring, and whoever joins,
    must still wait for them (the pooling reads the slot's sums on another stream)."""
    p = Layers(lib)
    assert p.run(1, one_side) == B.ASL_OK and p.run(0, one_side) == B.ASL_OK
    at = len(p.order()[0])
    if isinstance(fail, str):
        lib.fake_fail(fail.encode(), 1)
        assert p.run(1, one_side) == B.ASL_ERR_CUDA
    else:
        assert p.run(1, one_side, **fail) == B.ASL_ERR_INVALID
    names, _, _ = p.order()
    left = set(range(at, len(names)))
    assert names[at:] == issued
    assert p.lib.asl_run_join(p.ctx, 109) == B.ASL_OK
    assert left <= p.order()[2][109]
    nxt = len(names)
    assert p.run(1, one_side) == B.ASL_OK
    names, before, _ = p.order()
    assert names[nxt:] == ["score", "pool", "rank", "topk", "compact"]
    assert left <= before[nxt]
    p.close()


def test_layers_in_order(lib):
    """Three good layers: a step follows what it reads, and a slot's scoring what read the slot two layers ago."""
    p = Layers(lib)
    for slot in (0, 1, 0):
        assert p.run(slot) == B.ASL_OK
    names, before, _ = p.order()
    assert names == ["score", "pool", "rank", "topk", "compact"] * 3
    for l in range(3):
        i = 5 * l
        assert i in before[i + 1] and i + 1 in before[i + 2] and i + 1 in before[i + 3] and i + 3 in before[i + 4]
    assert {1, 2, 3, 4} <= before[10] and not {6, 7, 8, 9} & before[10]
    p.close()


def test_a_context_keeps_to_its_device(lib):
    """The events belong to the context's device, whichever was current when the first layer was run."""
    lib.cudaSetDevice(0)
    p = Layers(lib)
    assert p.run(0) == B.ASL_OK and lib.fake_device() == 0
    p.close()


@pytest.mark.parametrize("nth", [1, 3, 6])
def test_events_that_cannot_be_made(lib, nth):
    """No context, and nothing left behind, where one of its events cannot be made."""
    alive, ctx = lib.fake_alive(), C.c_void_p()
    lib.fake_fail(b"event", nth)
    assert lib.asl_create(C.byref(ctx), 1) == B.ASL_ERR_CUDA
    assert not ctx.value and lib.fake_alive() == alive
