"""What the C ABI's host code does with streams, failed calls and void states, seen on
a CUDA runtime of host memory (fake_cuda.cpp): no GPU, and no GPU fault, is needed."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1511_02155_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))
SIDE = ctypes.c_void_p(7)  # a stream that is not ordered with the default one
N = (40, 30)
dp = ctypes.POINTER(ctypes.c_double)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    if not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        cuda = "/usr/local/cuda/include"
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda, "-x", "c++",
                    os.path.join(_build.CSRC, "tlbm_api.cu"), os.path.join(HERE, "fake_cuda.cpp"), "-o", out], check=True)
    f = ctypes.CDLL(out)
    f.fake_log.restype = f.tlbm_last_error.restype = f.tlbm_batch_last_error.restype = ctypes.c_char_p
    d = ctypes.c_double
    f.tlbm_create.argtypes = [ctypes.POINTER(ctypes.c_void_p)] + [ctypes.c_int] * 4 + [dp, d, d, d, d, dp, ctypes.c_void_p,
                                                                                      ctypes.c_int, ctypes.c_void_p]
    f.tlbm_step.argtypes = [ctypes.c_void_p, ctypes.c_int64]
    f.tlbm_batch_step.argtypes = [ctypes.c_void_p, ctypes.c_int64]
    f.tlbm_destroy.restype = f.tlbm_batch_destroy.restype = None
    f.tlbm_state_bytes.restype = ctypes.c_size_t
    f.tlbm_set_gamma.argtypes = [ctypes.c_void_p, d, d]
    f.tlbm_get_state.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t]
    f.tlbm_adjoint_c3_misfit.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_int, dp, dp, dp, dp, dp]
    f.fake_fail.argtypes = [ctypes.c_char_p, ctypes.c_int]
    return f


def _create(lib, solid=True, precision=1):
    mask = np.zeros(N[0] * N[1], np.uint8)
    mask[:N[0]] = 1
    t = ctypes.c_void_p()
    rc = lib.tlbm_create(ctypes.byref(t), 9, *N, 1, (ctypes.c_double * 3)(0.01, 0.02, 0.03), 1.0, 1.0, 0.1, 0.1, None,
                         mask.ctypes.data if solid else None, precision, SIDE)
    return rc, t


@pytest.fixture
def fake(lib):
    lib.fake_reset()
    lib.fake_items(0, 5)
    yield lib
    lib.fake_reset()


def _steps(lib, t):
    """What a step saw, run when only the engine's own stream is waited for."""
    assert lib.tlbm_step(t, 1) == 0
    out = (ctypes.c_double * 3)()
    lib.tlbm_step_mass(t, out)
    return [s for s in lib.fake_log().decode().splitlines() if s.startswith("step")][-1]


def test_work_items_are_there_before_the_first_step(fake):
    rc, t = _create(fake)
    assert rc == 0
    assert _steps(fake, t) == "step: 5 items of tile 0"
    fake.fake_items(2 + 256 * 7, 9)
    assert fake.tlbm_set_tile(t, 2, 7) == 0
    assert _steps(fake, t) == f"step: 9 items of tile {2 + 256 * 7}"
    fake.tlbm_destroy(t)
    assert fake.fake_allocations() == 0


@pytest.mark.parametrize("call", [b"cudaMalloc", b"cudaMemcpy", b"cudaMemcpyAsync", b"cudaStreamSynchronize"])
def test_a_failed_upload_of_work_items_leaves_one_grid(fake, call):
    """Every step after it runs on the lattice's one grid; nothing is left allocated."""
    rc, t = _create(fake)
    assert rc == 0
    for nth in range(1, 4):
        tile = 256 * (6 + nth)
        fake.fake_items(tile, 9)
        before = fake.fake_allocations()
        fake.fake_fail(call, nth)
        failed = fake.tlbm_set_tile(t, 0, 6 + nth) != 0
        fake.fake_fail(b"", 0)
        assert _steps(fake, t) == ("step: one grid" if failed else f"step: 9 items of tile {tile}")
        assert fake.fake_allocations() == before + (0 if failed else 1)
        assert fake.tlbm_set_tile(t, 0, 0) == 0
    fake.tlbm_destroy(t)
    assert fake.fake_allocations() == 0


@pytest.mark.parametrize("capture", [1, 2])
def test_work_items_outlive_a_change_of_tile(fake, capture):
    """Steps captured at one tile may be replayed at any time later: their items stay,
    and a tile that was chosen before needs no call that a capture forbids."""
    rc, t = _create(fake)
    assert rc == 0
    tile = 2 + 256 * 7
    fake.fake_items(tile, 9)
    assert fake.tlbm_step(t, 1) == 0  # on the stream, not run yet: it holds the items of tile 0
    late = fake.fake_allocations()
    assert fake.tlbm_set_tile(t, 2, 7) == 0
    assert fake.fake_allocations() == late + 1  # and those are still allocated
    fake.fake_capturing(capture)
    assert fake.tlbm_set_tile(t, 0, 0) == 0 and fake.tlbm_step(t, 1) == 0
    assert fake.tlbm_set_tile(t, 2, 7) == 0 and fake.tlbm_step(t, 1) == 0
    fake.fake_items(256 * 3, 4)
    assert fake.tlbm_set_tile(t, 0, 3) == 0 and fake.tlbm_step(t, 1) == 0
    fake.fake_capturing(0)
    assert _steps(fake, t) == f"step: 4 items of tile {256 * 3}"
    assert fake.fake_log().decode().splitlines() == [
        "step: 5 items of tile 0", "step: 5 items of tile 0", f"step: 9 items of tile {tile}", "step: one grid",
        f"step: 4 items of tile {256 * 3}"]
    fake.tlbm_destroy(t)
    assert fake.fake_allocations() == 0


def test_kept_work_items_are_bounded(fake):
    rc, t = _create(fake)
    assert rc == 0
    cap = fake.tlbm_state_bytes(t) // 16 + 65536
    seen = set()
    for chunk in range(1, 41):
        fake.fake_items(256 * chunk, cap // 16 // 8)
        assert fake.tlbm_set_tile(t, 0, chunk) == 0
        seen.add(_steps(fake, t).split(" of ")[0])
        assert fake.fake_allocations() < 2 + 9
    assert seen == {f"step: {cap // 16 // 8} items", "step: one grid"}
    fake.tlbm_destroy(t)


def test_no_batched_step_after_a_failed_build(fake):
    """A build that fails half-way has replaced work items that the descriptors name: the
    batch builds again before it steps, whatever call had failed."""
    engines = [_create(fake)[1] for _ in range(2)]
    b = ctypes.c_void_p()
    assert fake.tlbm_batch_create(ctypes.byref(b), (ctypes.c_void_p * 2)(*engines), 2) == 0
    assert fake.tlbm_batch_step(b, 1) == 0
    fake.fake_build_fails(3)  # set_tile's own, and its return to the tile before; then the next step's
    assert fake.tlbm_batch_set_tile(b, 0, 7) != 0
    assert fake.tlbm_batch_step(b, 1) != 0
    assert fake.tlbm_batch_step(b, 1) == 0
    assert fake.fake_log().decode().split("\n") == [
        "batch build", "batch step", "batch build", "batch build", "batch build", "batch build", "batch step", ""]
    fake.tlbm_batch_destroy(b)
    for t in engines:
        fake.tlbm_destroy(t)


def _reads(fake, t):
    """Status of every call that returns data of the state."""
    n = N[0] * N[1]
    a = np.zeros(3 * 9 * n)
    p = a.ctypes.data_as(dp)
    size = fake.tlbm_state_bytes(t)
    raw = ctypes.create_string_buffer(size)
    return {"fields": fake.tlbm_fields(t, p, None, None, None, None), "mass": fake.tlbm_mass(t, p),
            "step_mass": fake.tlbm_step_mass(t, p), "populations": fake.tlbm_get_populations(t, p),
            "box": fake.tlbm_get_populations_box(t, 0, 0, 0, 1, 1, 1, p), "state": fake.tlbm_get_state(t, raw, size)}


def test_every_read_of_a_void_state_says_so(fake):
    rc, t = _create(fake, solid=False)
    assert rc == 0
    one = np.ones(N[0] * N[1]).ctypes.data_as(dp)
    nothing = (t, one, one, one, None, None, None)
    assert fake.tlbm_init_fields(*nothing) == 0
    assert fake.tlbm_step(t, 2) == 0 and set(_reads(fake, t).values()) == {0}
    fake.fake_flag(2)
    assert fake.tlbm_step(t, 1) == 0
    fake.fake_flag(0)
    assert fake.tlbm_step(t, 1) == 0  # a later step does not make it whole
    assert set(_reads(fake, t).values()) == {6}  # TLBM_ERR_TIMEOUT
    assert fake.tlbm_init_fields(*nothing) == 0 and set(_reads(fake, t).values()) == {0}
    fake.fake_flag(1)  # a non-finite total is step_mass's to report, as before
    assert fake.tlbm_step(t, 1) == 0
    assert {k: v for k, v in _reads(fake, t).items() if v} == {"step_mass": 5}
    fake.tlbm_destroy(t)


@pytest.mark.parametrize("flag,status", [(0, 0), (2, 6), (3, 6)])
def test_a_gradient_from_a_void_state_says_so(fake, flag, status):
    rc, t = _create(fake, solid=False)
    assert rc == 0
    one = np.ones(N[0] * N[1]).ctypes.data_as(dp)
    assert fake.tlbm_init_fields(t, one, one, one, None, None, None) == 0
    fake.fake_flag(flag)
    loss, out = ctypes.c_double(), (ctypes.c_double * 3)()
    assert fake.tlbm_adjoint_c3_misfit(t, 3, 2, one, ctypes.byref(loss), out, out, None) == status
    fake.tlbm_destroy(t)


def test_no_exception_leaves_the_c_entries(fake):
    """Host memory that runs out is TLBM_ERR_OOM, with nothing left behind."""
    oom = 4
    rc, t = _create(fake)
    rc2, t2 = _create(fake)
    assert rc == rc2 == 0
    one = np.ones(N[0] * N[1]).ctypes.data_as(dp)
    assert fake.tlbm_init_fields(t, one, one, one, None, None, None) == 0
    b = ctypes.c_void_p()
    assert fake.tlbm_batch_create(ctypes.byref(b), (ctypes.c_void_p * 1)(t2), 1) == 0
    held = fake.fake_allocations()
    fake.fake_throws(1)
    assert _create(fake)[0] == oom and b"memory" in fake.tlbm_last_error(None)
    none = ctypes.c_void_p()
    assert fake.tlbm_batch_create(ctypes.byref(none), (ctypes.c_void_p * 1)(t), 1) == oom and not none.value
    fake.fake_items(256 * 9, 3)
    loss, out = ctypes.c_double(), (ctypes.c_double * 3)()
    assert fake.tlbm_adjoint_c3_misfit(t, 3, 2, one, ctypes.byref(loss), out, out, None) == oom
    assert fake.tlbm_set_tile(t, 0, 9) == oom
    assert fake.tlbm_step(t, 1) == oom and b"memory" in fake.tlbm_last_error(t)
    assert fake.tlbm_launches_per_step(t) == -1
    assert fake.tlbm_batch_step(b, 1) == oom and b"memory" in fake.tlbm_batch_last_error(b)
    assert fake.tlbm_batch_set_tile(b, 0, 9) == oom
    assert fake.tlbm_batch_autotune(b, 1, None, None) == oom
    fake.fake_throws(0)
    assert fake.fake_allocations() == held
    assert fake.tlbm_batch_step(b, 1) == 0  # builds again first
    assert _steps(fake, t) == "step: one grid"
    fake.tlbm_batch_destroy(b)
    fake.tlbm_destroy(t)
    fake.tlbm_destroy(t2)
    assert fake.fake_allocations() == 0
