"""Which lattices and tiles the fused step takes: its dispatch rules compiled for the
host, against the rule that a plain tile and chunk by device fill give."""
import ctypes
import itertools
import os
import subprocess

import pytest

from paper_1511_02155_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))
SMS = 152


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("rules") / "librules.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-O1", "-shared", "-Xcompiler",
                    "-fPIC", os.path.join(HERE, "host_rules.cu"), "-o", out, "-cudart", "static"], check=True)
    lib = ctypes.CDLL(out)
    lib.rule_blocks.restype = ctypes.c_longlong
    return lib


def _plain_fits(Q, prec, shape, solid, coupling, chunk):
    """Whether the sums of plain tiles (rows of 128; 32x4, in double 16x8 or 16x4) fit the
    scratch at a given chunk, or at 64 (D3Q19: 16) halved until the device is full."""
    nx, ny, nz = shape
    if Q == 9:
        tx, ty, nb, nm = 128, 1, 1, ny
    else:
        tx, ty, nb, nm = (16, 4 if solid or coupling else 8, ny, nz) if prec == 0 else (32, 4, ny, nz)
    cols = -(-nx // tx) * -(-nb // ty)
    mc = chunk
    if mc == 0:
        mc = 64 if Q == 9 else 16
        while mc > 4 and cols * -(-nm // mc) < 4 * SMS:
            mc //= 2
    mc = min(mc, nm)
    return cols * -(-nm // mc) <= max(nx * ny * nz // 64 + 1, 1216)


ROWS = [1, 2, 3, 31, 32, 33, 63, 64, 65, 127, 129, 500, 1216, 5000, 38912, 38913, 50000, 77823, 77825, 300000]


@pytest.mark.parametrize("chunk", [0, 1, 7, 64])
@pytest.mark.parametrize("coupling,solid", [(0, 0), (0, 1), (1, 0)])
@pytest.mark.parametrize("Q,prec", [(9, 0), (9, 1), (19, 0), (19, 1)])
def test_every_lattice_that_plain_tiles_take_is_taken(rules, Q, prec, coupling, solid, chunk):
    sizes = [(x, y, 1) for x, y in itertools.product(ROWS, ROWS)] if Q == 9 else \
        [(x, y, z) for x, y, z in itertools.product(ROWS[::3], ROWS[::4], ROWS[1::4])]
    lost = [s for s in sizes if s[0] * s[1] * s[2] < 4e7 and _plain_fits(Q, prec, s, solid, coupling, chunk)
            and rules.rule_blocks(Q, prec, *s, solid, coupling, 256 * chunk, SMS) < 0]
    assert not lost, lost[:10]


@pytest.mark.parametrize("nx,ny", [(517, 391), (389, 500), (1000, 701)])
def test_a_short_clean_run_does_not_set_the_chunk_of_all_blocks(rules, nx, ny):
    """Planes near solid nodes march as far as they would without one gap among them."""
    alone = rules.rule_longest_dirty(nx, ny, 0, SMS)
    for clean in (9, 12):  # five and eight planes that are two nodes from the others
        assert abs(rules.rule_longest_dirty(nx, ny, clean, SMS) - alone) <= 1
