"""GPU parity of the marching kernels at the edges of their tiles and rules.

Every case takes one step from populations that the engine itself holds (rounded
to its storage) and compares with the FP64 oracle's step from the same numbers.
Bounds, per population:
- FP64 storage: 1e-13 (a few hundred operations on values below 1);
- FP32 storage: 2e-6, the rounding of one step used by the full-size tests;
- 16-bit storage: 2e-6 plus half a unit in the last place of the stored value,
  |x| 2^-11 (FP16) or |x| 2^-8 (BF16), at the largest moving deviation.
"""
import math

import numpy as np
import pytest

import oracle
import paper_1511_02155_gb300 as tl
from paper_1511_02155_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

KAPPA = (0.012, 0.02, 0.016)
H = (0.0005, -0.0004, 0.0003)
HALF_ULP = {"fp16": 2.0 ** -11, "bf16": 2.0 ** -8}


def _weights(Q):
    if Q == 9:
        return np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
    return np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def _one_step(Q, shape, precision, solid=None, tile=(0, 0), forcing=False, steps=1):
    """Largest error of `steps` steps against the oracle, and the bound for one."""
    nx, ny, nz = shape
    sh = (ny, nx) if Q == 9 else (nz, ny, nx)
    C = W.spinodal(sh, seed=nx + ny + nz, amp=0.2)
    fields = W.to_aux(*C)
    if solid is not None:
        for a in fields:
            a[solid != 0] = 0.0
    h = H if solid is not None else (0.0, 0.0, 0.0)
    eng = tl.TernaryLB(Q, nx, ny, nz, KAPPA, 1.0, 0.8, 0.1, 0.1, h, None if solid is None else solid.reshape(-1), precision)
    if forcing:
        eng.set_coupling("forcing")
    eng.set_tile(*tile)
    rng = np.random.default_rng(5)
    u = [rng.uniform(-0.02, 0.02, sh) for _ in range(3)]
    if Q == 9:
        u[2][:] = 0.0
    eng.init_fields(*fields, u=u)
    eng.step(2)  # away from equilibrium
    P = eng.get_populations()
    p = oracle.make_params(Q, nx, ny, nz, KAPPA, 1.0, 0.8, 0.1, 0.1, h)
    f, g, k = (np.ascontiguousarray(P[s]) for s in range(3))
    before = eng.mass()
    eng.step(steps)
    if forcing:
        oracle.step_guo(p, f, g, k, steps)
    else:
        oracle.step(p, f, g, k, steps, *(() if solid is None else (solid.reshape(-1),)))
    got = eng.get_populations()
    want = np.stack([a.reshape(Q, -1) for a in (f, g, k)])
    if solid is not None:
        got, want = got[:, :, solid.reshape(-1) == 0], want[:, :, solid.reshape(-1) == 0]
    err = np.abs(got - want).max()
    if steps == 1:
        assert np.allclose(eng.step_mass(), before, rtol=0, atol=1e-9 * max(1.0, np.prod(sh)))
    eng.close()
    bound = {"fp64": 1e-13, "fp32": 2e-6}.get(precision, 2e-6)
    if precision in HALF_ULP:
        moving = want[:, 1:].copy()
        moving[0] -= _weights(Q)[1:, None]
        bound += HALF_ULP[precision] * np.abs(moving).max()
        # the rest population closes the node's moment over Q - 1 rounded values
        bound *= Q - 1
    return err, bound


# D3Q19 chunks of 32 nodes: one partial, one whole, a tail of one, of two, an odd
# tail; rows fewer than, equal to and one more than a tile; one plane
@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 2), (31, 4, 3), (32, 5, 1), (33, 8, 4), (34, 9, 5), (65, 2, 7),
                                   (96, 13, 6)])
def test_periodic_d3q19_at_tile_edges(shape, precision):
    err, bound = _one_step(19, shape, precision)
    assert err <= bound, (err, bound)


@pytest.mark.parametrize("chunk", [1, 3, 7])
def test_periodic_d3q19_chunks(chunk):
    err, bound = _one_step(19, (40, 7, 11), "fp32", tile=(0, chunk))
    assert err <= bound, (err, bound)


# rows narrower and wider than one-warp rows and than 128, few and many planes
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (31, 5, 1), (32, 64, 1), (33, 9, 1), (129, 40, 1)])
def test_periodic_d2q9_small_lattices(shape, precision):
    err, bound = _one_step(9, shape, precision)
    assert err <= bound, (err, bound)


def _mask(Q, shape, kind):
    """Solid nodes that leave clean, dirty and all-solid blocks in many places."""
    nx, ny, nz = shape
    s = np.zeros((ny, nx) if Q == 9 else (nz, ny, nx), np.uint8)
    up = s  # march axis first
    if kind == "walls":
        up[:2] = 1
        up[-1] = 1
    elif kind == "block":
        up[:9] = 1
        up[4:9, ..., nx // 4:nx // 2] = 0
        up[-1] = 1
    elif kind == "speck":  # one node at a tile's corner, and one at the periodic edge
        up[s.shape[0] // 2, ..., 31] = 1
        up[0, ..., 0] = 1
    elif kind == "porous":
        up[np.random.default_rng(3).random(s.shape) < 0.03] = 1
    return s


@pytest.mark.parametrize("precision,tile", [("fp32", (0, 0)), ("fp32", (2, 5)), ("fp32", (3, 16)), ("fp16", (0, 0)),
                                            ("fp64", (0, 0))])
@pytest.mark.parametrize("kind", ["walls", "block", "speck", "porous"])
@pytest.mark.parametrize("shape", [(40, 30, 1), (161, 90, 1), (300, 48, 1)])
def test_solid_d2q9_clean_and_dirty_blocks(shape, kind, precision, tile):
    err, bound = _one_step(9, shape, precision, _mask(9, shape, kind), tile)
    assert err <= bound, (err, bound)


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("kind", ["walls", "speck"])
def test_solid_d3q19_with_a_launch_for_clean_blocks(kind, precision):
    shape = (98, 165, 40)  # columns enough for clean blocks to fill the device
    solid = _mask(19, shape, kind)
    err, bound = _one_step(19, shape, precision, solid)
    assert err <= bound, (err, bound)
    eng = tl.TernaryLB(19, *shape, KAPPA, solid=solid.reshape(-1), precision=precision)
    assert eng.launches_per_step == 3
    eng.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("Q,shape", [(19, (33, 9, 5)), (19, (31, 7, 2)), (19, (2, 1, 1)), (9, (129, 6, 1)), (9, (5, 3, 1))])
def test_forcing_at_tile_edges(Q, shape, precision):
    err, bound = _one_step(Q, shape, precision, forcing=True)
    assert err <= bound, (err, bound)


@pytest.mark.parametrize("Q,shape,precision,tile", [
    # chunks of one plane whose sums fit the scratch (max(1216, N / 64 + 1) blocks) only on wider tiles
    (9, (128, 600, 1), "fp64", (0, 1)), (9, (33, 1000, 1), "fp64", (0, 1)), (9, (64, 640, 1), "fp64", (0, 1)),
    (19, (64, 1, 1800), "fp32", (2, 1)), (19, (5, 5, 1216), "fp16", (1, 1))])
def test_given_chunks_of_one_plane_still_fit_the_scratch(Q, shape, precision, tile):
    err, bound = _one_step(Q, shape, precision, tile=tile)
    assert err <= bound


def test_batch_of_double_members_with_chunks_of_one_plane():
    """One member's sums fit only on rows of 128, the other's on either: three steps to rounding."""
    def engines():
        out = []
        for nx, ny in ((128, 600), (64, 40)):
            eng = tl.TernaryLB(9, nx, ny, 1, KAPPA, precision="fp64")
            eng.init_fields(*W.to_aux(*W.spinodal((ny, nx), seed=nx, amp=0.1)))
            out.append(eng)
        return out

    alone, members = engines(), engines()
    batch = tl.TernaryBatch(members)
    batch.set_tile(0, 1)
    batch.step(3)
    for x, y in zip(alone, members):
        x.set_tile(0, 1)
        x.step(3)
        assert np.abs(x.get_populations() - y.get_populations()).max() <= 3e-13
    batch.close()
    for e in alone + members:
        e.close()


def test_many_steps_in_one_call_equal_single_steps():
    """Steps overlap their launches; a call of n steps gives the bits of n calls."""
    for Q, shape, solid in ((9, (70, 50, 1), None), (9, (70, 50, 1), "walls"), (19, (40, 9, 8), None)):
        s = None if solid is None else _mask(Q, shape, solid)
        states = []
        for split in (False, True):
            eng = tl.TernaryLB(Q, *shape, KAPPA, h=H if s is not None else (0, 0, 0),
                               solid=None if s is None else s.reshape(-1), precision="fp32")
            C = W.spinodal((shape[1], shape[0]) if Q == 9 else shape[::-1], seed=4, amp=0.1)
            f = W.to_aux(*C)
            if s is not None:
                for a in f:
                    a[s != 0] = 0.0
            eng.init_fields(*f)
            for _ in range(9 if split else 1):
                eng.step(1 if split else 9)
                if split:
                    eng.step_mass()
            states.append((eng.get_populations(), eng.step_mass()))
            eng.close()
        assert np.array_equal(states[0][0], states[1][0]) and np.array_equal(states[0][1], states[1][1])


@pytest.mark.parametrize("nx", [38913, 50000])
def test_a_single_row_in_double(nx):
    """Rows of 32 nodes would have more blocks than the scratch has sums, at any chunk."""
    err, bound = _one_step(9, (nx, 1, 1), "fp64")
    assert err <= bound
    states = []
    for batched in (False, True):
        engines = []
        for n in (nx, 40):
            eng = tl.TernaryLB(9, n, 1, 1, KAPPA, precision="fp64")
            eng.init_fields(*W.to_aux(*W.spinodal((1, n), seed=n, amp=0.1)))
            engines.append(eng)
        if batched:
            with tl.TernaryBatch(engines) as b:
                b.step(3)
        else:
            for e in engines:
                e.step(3)
        states.append([e.get_populations() for e in engines])
        for e in engines:
            e.close()
    for a, b in zip(*states):
        assert np.abs(a - b).max() <= 3e-13


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("kind", ["walls", "speck", "porous_floor"])
def test_solid_d3q19_steps_side_by_side_equal_one_grid(kind, precision):
    """Clean and dirty blocks in two launches against the solid-aware blocks alone (too few
    clean columns for two launches at one chunk a column): many steps, the same bits."""
    shape = (98, 165, 40)
    if kind == "porous_floor":
        solid = _mask(19, shape, "walls")
        solid[2:5][np.random.default_rng(8).random(solid[2:5].shape) < 0.2] = 1
    else:
        solid = _mask(19, shape, kind)
    f = W.to_aux(*W.spinodal(shape[::-1], seed=2, amp=0.1))
    for a in f:
        a[solid != 0] = 0.0
    out = []
    for chunk, launches in ((0, 3), (4096, 2)):
        eng = tl.TernaryLB(19, *shape, KAPPA, h=H, solid=solid.reshape(-1), precision=precision)
        eng.set_tile(0, chunk)
        assert eng.launches_per_step == launches
        eng.init_fields(*f)
        eng.step(41)
        eng.step(1)
        eng.step(18)
        out.append(eng.get_populations())
        eng.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("Q,shape,kind,tile", [
    (9, (300, 48, 1), "walls", (0, 0)), (9, (161, 90, 1), "porous", (0, 0)), (9, (300, 48, 1), "block", (0, 7)),
    (9, (300, 48, 1), "walls", (2, 0)), (9, (161, 90, 1), "block", (3, 5)), (19, (98, 165, 40), "walls", (0, 0)),
    (19, (98, 165, 40), "speck", (0, 9))])
def test_checked_steps_take_the_work_items(Q, shape, kind, tile):
    """Clean and dirty blocks checked: nothing recorded, the unchecked step's bits."""
    solid = _mask(Q, shape, kind)
    f = W.to_aux(*W.spinodal(shape[1::-1] if Q == 9 else shape[::-1], seed=6, amp=0.1))
    for a in f:
        a[solid != 0] = 0.0
    out = []
    for checked in (False, True):
        eng = tl.TernaryLB(Q, *shape, KAPPA, h=H, solid=solid.reshape(-1), precision="fp32")
        eng.set_tile(*tile)
        launches = eng.launches_per_step
        eng.set_bounds_check(checked)
        if Q == 19:
            assert eng.launches_per_step == launches == 3
        eng.init_fields(*f)
        eng.step(6)
        assert eng.bounds_check_word() == 0
        out.append(eng.get_populations())
        eng.close()
    assert np.array_equal(out[0], out[1])


def test_captured_steps_replay_with_solid_nodes():
    """tlbm_step under stream capture, a change of tile between capture and replay, and a
    capture begun after one."""
    for Q, shape in ((9, (300, 90, 1)), (19, (98, 165, 40))):
        solid = _mask(Q, shape, "walls")
        f = W.to_aux(*W.spinodal(shape[1::-1] if Q == 9 else shape[::-1], seed=6, amp=0.1))
        for a in f:
            a[solid != 0] = 0.0
        side = torch.cuda.Stream()
        want = tl.TernaryLB(Q, *shape, KAPPA, h=H, solid=solid.reshape(-1), precision="fp32")
        with torch.cuda.stream(side):
            eng = tl.TernaryLB(Q, *shape, KAPPA, h=H, solid=solid.reshape(-1), precision="fp32")
        for e in (want, eng):
            e.init_fields(*f)
            e.step(2)
        graphs = []
        for tile in ((0, 0), (2, 5)):
            eng.set_tile(*tile)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side):
                eng.step(2)
            graphs.append(g)
        eng.set_tile(3, 9)
        with torch.cuda.stream(side):
            for k in (0, 1, 0, 0, 1):
                graphs[k].replay()
        side.synchronize()
        want.step(10)
        assert np.array_equal(eng.get_populations(), want.get_populations())
        want.close()
        eng.close()


@pytest.mark.parametrize("forcing", [False, True])
@pytest.mark.parametrize("chunk", [0, 64])
def test_totals_of_d3q19_fp32_are_double_sums(chunk, forcing):
    """Values of one column whose sum has 52 bits, and so is exact in double in any order;
    pairs of floats round it."""
    shape, rng = (4, 4, 64), np.random.default_rng(9)
    v = np.concatenate([1 + 2.0 ** -23 * rng.integers(1, 2 ** 22, 32), 2.0 ** -45 * rng.integers(2 ** 19, 2 ** 20, 32)])
    v = v.astype(np.float32).astype(np.float64)
    eng = tl.TernaryLB(19, *shape, KAPPA, precision="fp32")
    if forcing:
        eng.set_coupling("forcing")
    eng.set_tile(0, chunk)
    one, zero = np.ones(eng.N), np.zeros(eng.N)
    eng.init_fields(one, zero, zero)
    P = eng.get_populations()
    P[1:] = 0.0
    for s, sign in ((1, -1.0), (2, 1.0)):  # rest populations phi and psi of the column at (2, 1)
        P[s, 0].reshape(64, 4, 4)[:, 1, 2] = sign * v
    eng.set_populations(P)
    eng.step(1)
    m = eng.step_mass()
    assert m[2] == math.fsum(v) and m[1] == -math.fsum(v)
    eng.close()
