"""The kernels with bulk copies where the engine never takes them: a wait that runs out."""
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
