"""The library's host code against a CUDA runtime without a GPU (``host/fake_runtime.cpp``): what it does
between the calls of a user and the launches, where a mistake would fault or hang a real device or needs a
second one to show."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2309_08068_gb300 import build as lbm_build
from paper_2309_08068_gb300 import lbm

HERE = os.path.dirname(os.path.abspath(__file__))
SINGLE, RING, TILED, LINE, BATCHED = range(5)
MM, HV = 0, 1
STREAM = 0x1000  # any stream but the legacy one: the fake runtime tells them apart by value


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    lbm_build.build(force=not all(os.path.exists(o) for o in lbm_build.objects()))
    so = str(tmp_path_factory.mktemp("host") / "liblbm_host.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-std=c++17", "-Wl,-Bsymbolic", "-Wl,-z,defs",
                    "-I", os.path.join(os.path.dirname(os.path.dirname(lbm_build.nvcc())), "include"), "-o", so,
                    os.path.join(HERE, "host", "fake_runtime.cpp"), *lbm_build.objects()], check=True)
    L = ctypes.CDLL(so)
    L.lbm_last_error.restype = ctypes.c_char_p
    L.lbm_last_error.argtypes = [ctypes.c_void_p]
    L.lbm_time.restype, L.lbm_time.argtypes = ctypes.c_int64, [ctypes.c_void_p]
    L.lbm_step.argtypes = [ctypes.c_void_p, ctypes.c_int]
    L.lbm_step_fusion_active.argtypes = [ctypes.c_void_p]
    L.lbm_set_step_fusion.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    L.lbm_batch_create.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    L.lbm_batch_step.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    L.lbm_batch_destroy.argtypes = [ctypes.c_void_p]
    L.lbm_adjoint.argtypes = [ctypes.c_void_p] + [ctypes.c_int] * 4 + [ctypes.c_void_p] * 3 + [ctypes.c_int]
    L.lbm_set_source.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    L.lbm_clear_sources.argtypes = L.lbm_destroy.argtypes = [ctypes.c_void_p]
    L.fake_reset()
    return L


class Context:
    """A context of the C ABI on the fake runtime."""

    def __init__(self, lib, model, shape, mode=1, eps_r=None, storage=0, stream=STREAM):
        self.lib, self.h = lib, ctypes.c_void_p()
        media = None
        if eps_r is not None:
            self.eps = np.ascontiguousarray(eps_r, np.float32)
            media = ctypes.byref(lbm._Media(self.eps.ctypes.data, None, None, 0))
        opts = lbm._Options(storage, ctypes.c_void_p(stream), 0, 0.0, 0.0, 0.0, 0)
        assert lib.lbm_create(model, *shape, media, ctypes.byref(opts), ctypes.byref(self.h)) == 0
        assert lib.lbm_set_step_fusion(self.h, mode, 0) == 0

    def add_current(self, cells):
        cells = np.asarray(cells, np.int64)
        w = np.ones(3 * cells.size, np.float32)
        fn = lbm._TimeFn(lbm.FN_KINDS["const"], 1.0, 0.0, 0.0, None, 0)
        s = lbm._Source(lbm.SRC_KINDS["current"], cells.size, cells.ctypes.data, w.ctypes.data, (ctypes.c_float * 3)(),
                        (ctypes.c_float * 3)(), fn)
        assert self.lib.lbm_set_source(self.h, ctypes.byref(s)) == 0

    def step(self, n):
        rc = self.lib.lbm_step(self.h, n)
        return rc, self.lib.lbm_last_error(self.h).decode()

    def close(self):
        assert self.lib.lbm_destroy(self.h) == 0


@pytest.mark.parametrize("model,shape,mode,kind", [
    (HV, (80, 80, 80), 1, TILED), (MM, (96, 96, 96), 1, TILED), (HV, (16, 16, 3), 3, TILED),
    (HV, (256, 256, 16), 1, RING), (MM, (256, 160, 8), 2, RING), (MM, (1, 1, 500), 1, LINE), (HV, (24, 24, 24), 0, SINGLE)])
def test_uploads_have_arrived_before_the_launch_that_reads_them(lib, model, shape, mode, kind):
    """Media, source lists and the passes' lists are copied from pageable memory on the legacy stream, which
    the context's stream does not wait for: the host has to, before the next launch."""
    lib.fake_reset()
    n = int(np.prod(shape))
    eps = None if kind == RING and mode == 1 else 1.0 + np.arange(n) % 5
    c = Context(lib, model, shape, mode, eps)
    assert c.step(4)[0] == 0
    c.add_current([n // 2])
    assert c.step(4)[0] == 0
    assert lib.lbm_clear_sources(c.h) == 0
    assert c.step(4)[0] == 0
    assert lib.fake_launches(kind) > 0 and lib.fake_early_launches() == 0
    c.close()


@pytest.mark.parametrize("model,shape,mode", [(HV, (80, 80, 80), 1), (MM, (96, 96, 96), 1), (HV, (16, 16, 3), 3),
                                              (MM, (1, 1, 500), 1), (MM, (24, 24, 24), 1)])
def test_first_steps_may_be_captured(lib, model, shape, mode):
    """Building the tiled pass's lists does not break the capture of a context's first call, nor of the first
    after its sources changed, and the thread's capture mode is what it was."""
    lib.fake_reset()
    c = Context(lib, model, shape, mode)
    for _ in range(2):
        lib.fake_capture(1)
        assert c.step(4) == (0, "")
        assert not lib.fake_capture_broken()
        assert lib.fake_early_launches() == 0
        p = ctypes.c_void_p()
        assert lib.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(8)) != 0  # refused again
        lib.cudaGetLastError()
        lib.fake_capture(0)
        c.add_current([0, 1])
    c.close()


@pytest.mark.parametrize("model,shape,mode", [(HV, (80, 80, 80), 1), (MM, (16, 16, 3), 3), (HV, (1, 1, 500), 1),
                                              (MM, (1, 1, 30000), 1)])
@pytest.mark.parametrize("steps", [2, 3, 4, 5, 6, 7, 33, 56, 57, 58, 113, 1000])
def test_captured_calls_swap_the_buffers_as_single_steps_do(lib, model, shape, mode, steps):
    """So that a graph of an even number of steps can be replayed. Outside a capture a call takes as few passes
    or launches as it can."""
    lib.fake_reset()
    c = Context(lib, model, shape, mode)
    swaps = []
    for captured in (0, 1):
        before = sum(lib.fake_launches(k) for k in (SINGLE, RING, TILED, LINE))
        lib.fake_capture(captured)
        assert c.step(steps)[0] == 0
        lib.fake_capture(0)
        swaps.append(sum(lib.fake_launches(k) for k in (SINGLE, RING, TILED, LINE)) - before)
    assert swaps[1] % 2 == steps % 2 and swaps[0] <= swaps[1] <= swaps[0] + 1
    assert lib.lbm_time(c.h) == 2 * steps
    c.close()


def test_ring_passes_are_not_captured(lib):
    """Their blocks wait for flags that carry the pass's number, which a graph repeats: a replay's waits would
    find the flags of the one before."""
    lib.fake_reset()
    c = Context(lib, MM, (256, 160, 8), 2)
    lib.fake_capture(1)
    assert c.step(5) == (0, "") and not lib.fake_capture_broken()
    lib.fake_capture(0)
    assert lib.fake_launches(RING) == 0 and lib.fake_launches(SINGLE) == 5
    assert c.step(5)[0] == 0 and lib.fake_launches(RING) == 2
    c.close()


@pytest.mark.parametrize("storage,cells,kind", [("f24", 500, LINE), ("f24", 24000, LINE), ("f24", 24001, SINGLE),
                                                ("f24", 1000000, SINGLE), ("bf16", 1000000, LINE), ("f32", 1000000, LINE)])
def test_long_lines_of_24_bit_storage_step_singly(lib, storage, cells, kind):
    """Many steps per launch were up to twice as slow there as the launch per step that they replaced."""
    lib.fake_reset()
    c = Context(lib, MM, (1, 1, cells), storage=lbm.STORAGE[storage])
    assert c.step(8)[0] == 0
    assert [k for k in (SINGLE, LINE) if lib.fake_launches(k)] == [kind]
    c.close()


# (cells of each line, its steps), steps of a 16^3 lattice beside them, and which lines step on their own
@pytest.mark.parametrize("model,storage,lines,cube,alone", [
    (MM, "f32", [(500, 64)] * 6, 0, [1] * 6),                     # few lines and nothing else
    (MM, "f32", [(500, 64)] * 7, 0, [0] * 7),
    (MM, "f32", [(500, 64)] * 3, 64, [0] * 3),                    # the batched launches are needed anyway
    (HV, "f32", [(500, 64), (24000, 64)], 64, [0, 1]),            # long lines gain even so
    (HV, "f32", [(23999, 64)], 64, [0]),
    (MM, "f32", [(500, 640)] * 3, 10, [1] * 3),                   # ... but not for as many steps
    (MM, "f32", [(500, 640)] * 3, 321, [0] * 3),
    (MM, "f32", [(500, 64), (500, 1)], 0, [1, 0]),
    (MM, "bf16", [(500, 64)] * 4, 0, [1] * 4),
    (MM, "bf16", [(500, 64)] * 5, 0, [0] * 5),
    (HV, "f16", [(500, 64)] * 6, 0, [1] * 6),
    (HV, "f16", [(16384, 64), (24001, 64)], 0, [0, 0]),
    (HV, "f24", [(500, 64)], 0, [1]),
    (HV, "f24", [(500, 64)] * 2, 0, [0] * 2),
])
def test_lines_of_a_batch_step_on_their_own_where_that_is_faster(lib, model, storage, lines, cube, alone):
    lib.fake_reset()
    shapes = [(1, 1, n) for n, _ in lines] + ([(16, 16, 16)] if cube else [])
    steps = [s for _, s in lines] + ([cube] if cube else [])
    group = [Context(lib, model, s, storage=lbm.STORAGE[storage]) for s in shapes]
    b = ctypes.c_void_p()
    assert lib.lbm_batch_create((ctypes.c_void_p * len(group))(*[c.h for c in group]), len(group), ctypes.byref(b)) == 0
    assert lib.lbm_batch_step(b, (ctypes.c_int * len(steps))(*steps)) == 0
    launches = [lib.fake_launches(k) for k in (LINE, BATCHED)]
    batched = [s for s, own in zip(steps, alone + [0]) if not own]
    assert launches[1] == max(batched, default=0)
    own = [s for (_, s), a in zip(lines, alone) if a]
    assert sum(-(-s // 56) for s in own) <= launches[0] <= sum(-(-s // 32) for s in own)
    assert lib.lbm_batch_destroy(b) == 0
    for c in group:
        c.close()


@pytest.mark.parametrize("model,storage", [(HV, "f32"), (HV, "f16"), (MM, "f32"), (MM, "bf16")])
def test_tiled_pass_on_every_device(lib, model, storage):
    """The pass's shared memory has to be allowed on each device that runs it, not once per process."""
    shape = (16, 16, 8)
    eps = {"f32": None, "f16": 1.0 + np.arange(2048) % 5, "bf16": 1.0 + np.arange(2048) / 4096}[storage]
    for device in (0, 1, 0):
        lib.fake_reset()
        lib.fake_set_device(device)
        c = Context(lib, model, shape, 3, eps, lbm.STORAGE[storage])
        rc, msg = c.step(4)
        assert rc == 0, (device, msg)
        assert lib.fake_launches(TILED) == 2
        if storage == "f32" and model == MM:  # the recording pass of the adjoint
            loss = ctypes.c_double()
            assert lib.lbm_adjoint(c.h, 4, 2, 0, -1, ctypes.byref(loss), None, None, 0) == 0, (device, c.step(0)[1])
            assert lib.fake_launches(TILED) == 4
        c.close()


def test_tiled_pass_is_not_chosen_where_its_shared_memory_is_refused(lib):
    """Lattices step singly there; once it is allowed, new contexts take the pass."""
    lib.fake_reset()
    lib.fake_set_device(2)
    lib.fake_refuse_shared(1)
    for model, mode in ((HV, 1), (MM, 3)):
        c = Context(lib, model, (96, 96, 96), mode)
        assert lib.lbm_step_fusion_active(c.h) == 0
        assert c.step(3)[0] == 0 and lib.fake_launches(TILED) == 0
        c.close()
    assert lib.fake_launches(SINGLE) == 6
    lib.fake_refuse_shared(0)
    c = Context(lib, HV, (96, 96, 96))
    assert c.step(3)[0] == 0 and lib.fake_launches(TILED) == 1
    c.close()
