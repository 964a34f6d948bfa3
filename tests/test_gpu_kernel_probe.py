"""The kernels with bulk copies where the engine never takes them: a wait that runs out,
and checked steps that are told of a smaller buffer than they have."""
import ctypes
import os
import subprocess

import pytest

from paper_1511_02155_gb300 import _build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "libprobe.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-O3", "-shared", "-Xcompiler",
                    "-fPIC", os.path.join(HERE, "kernel_probe.cu"), "-o", out, "-cudart", "static"], check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("Q", [9, 19])
def test_a_wait_that_runs_out_ends_with_a_status(probe, Q):
    """Barriers that a missing warp never completes: the flag is raised, nothing is stored
    in the new state, and the kernel ends after its two limits of a second."""
    flag, stored, seconds = ctypes.c_int(-1), ctypes.c_longlong(-1), ctypes.c_double()
    assert probe.probe_late(Q, ctypes.byref(flag), ctypes.byref(stored), ctypes.byref(seconds)) == 0
    assert flag.value == 2
    assert stored.value == 0
    assert 1.0 <= seconds.value <= 10.0


# bytes of one plane of the probe's lattices: 9 rows (one) of two (seven) chunks
PLANE = {19: 9 * 2 * 57 * 128, 9: 7 * 27 * 128}


@pytest.mark.parametrize("Q", [9, 19])
@pytest.mark.parametrize("M0,M1,cut,code", [
    (2, 4, 0, 0),      # planes 0 .. 5 are read: nothing to record
    (2, 4, "2", 0),    # ... nor where the buffer ends behind plane 5
    (0, 2, "2", 1),    # planes 6 and 7, the periodic halo of plane 0, are beyond the end
    (2, 4, "2+", 1),   # the end lies inside a copy of plane 5
])
def test_checked_copies_stay_in_the_buffer_they_are_told_of(probe, Q, M0, M1, cut, code):
    """Every read is physically inside the populations; the checked step must see those
    that are outside the smaller extent it is given, plane offsets and lengths included."""
    n = {0: 0, "2": 2 * PLANE[Q], "2+": 2 * PLANE[Q] + 64}[cut]
    if cut == "2+" and Q == 19:
        n += PLANE[Q] - 4 * 2 * 57 * 128  # inside the fourth row, which the first tile reads
    elif cut == "2+":
        n += 2 * 27 * 128  # inside the fifth chunk, the x neighbours of the first tile
    word, size = ctypes.c_ulonglong(99), ctypes.c_longlong()
    assert probe.probe_check(Q, M0, M1, ctypes.c_longlong(n), ctypes.byref(word), ctypes.byref(size)) == 0
    assert word.value >> 56 == code
    if code:
        at = word.value & ((1 << 56) - 1)
        assert size.value - 27 * 128 * 3 < at < size.value + n
