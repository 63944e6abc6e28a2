"""Forms of a step that only large grids reach, bit for bit against another form of the same step: planes
of both phases on D2Q5 and D2Q9 with their stored populations, phi as pairs beside tiled U and theta in
3D under both block heights, and node-wise blocks of fewer warps."""
import numpy as np
import pytest

from paper_1602_07483_gb300 import lbpf, workloads

pytestmark = pytest.mark.gpu


def _init(sims):
    nx, ny, nz = sims[0].nx, sims[0].ny, sims[0].nz
    rng = np.random.default_rng(5)
    c = np.stack([rng.integers(0, n, 6) for n in (nx, ny, nz)], 1).astype(np.float64)
    r = rng.uniform(5.0, 12.0, 6)
    for s in sims:
        s.init_seed(c, r, -0.55, -0.3)


def _same(a, b, state):
    for x, y in zip(a.read_fields(), b.read_fields()):
        assert np.isfinite(x).all() and np.array_equal(x, y)
    if state:
        for x, y in zip(a.get_state(), b.get_state()):
            assert x is None or np.array_equal(x, y)


# beside a member with odd rows every member of a batch is tiled; alone, both phases run as planes
# (FP32 from 4.5 M nodes on), one chunk and many, ragged last tiles
@pytest.mark.parametrize("storage,shape,lattices", [("f32", (2202, 2050, 1), (5, 5, 9)), ("f32", (2202, 2050, 1), (9, 9, 0)),
                                                    ("f16", (1030, 1100, 1), (5, 9, 5)), ("f16", (130002, 9, 1), (9, 9, 9)),
                                                    ("bf16", (1030, 1100, 1), (5, 5, 9)), ("bf16", (62, 40000, 1), (9, 5, 5))])
def test_planes_equal_tiles_with_populations(storage, shape, lattices):
    p = workloads.base_params(kappa=100.0)
    shapes = [shape, (1101, 1100, 1)]
    batch = lbpf.Batch.create(shapes, lattices, [lbpf.make_params(storage, **p) for _ in shapes])
    alone = lbpf.Sim(shape, lattices, storage=storage, **p)
    _init([batch.sims[0], alone])
    _init([batch.sims[1]])
    batch.step(7)
    alone.step(7)
    _same(batch.sims[0], alone, state=True)
    batch.close()


# phi as pairs, U and theta as tiles with the block height compiled in (by = 8) and without (by = 5), against
# the one-launch step, whose phi is tiled too
@pytest.mark.parametrize("tiling", [(0, 0), (5, 0), (5, 17)])
def test_mixed_3d_step_equals_one_launch(tiling):
    shape, lattices = (202, 201, 200), (19, 19, 19)
    p = dict(workloads.base_params(kappa=100.0), aniso=1, eps1=-0.02, eps2=0.015, dt=0.01)
    a, b = (lbpf.Sim(shape, lattices, storage="f32", **p) for _ in range(2))
    _init([a, b])
    if tiling != (0, 0):
        a.set_tiling(*tiling)
    b.set_schedule("one_launch")
    assert a.step_launches == 3 and b.step_launches == 1
    a.step(8)
    b.step(8)
    _same(a, b, state=False)


# rows (2D) and planes (3D) shorter than a block take fewer warps; beside a wide member, whole blocks
@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("shape,wide,lattices", [((16, 700, 1), (400, 30, 1), (9, 5, 5)), ((33, 300, 1), (301, 30, 1), (9, 9, 0)),
                                                 ((90, 200, 1), (400, 30, 1), (5, 9, 5)), ((4, 4, 300), (40, 20, 9), (19, 19, 7)),
                                                 ((5, 7, 200), (41, 20, 9), (15, 7, 19)), ((1, 1, 50), (40, 20, 9), (19, 7, 7))])
def test_short_blocks_equal_whole_ones(storage, shape, wide, lattices):
    p = workloads.base_params(kappa=100.0)
    batch = lbpf.Batch.create([shape, wide], lattices, [lbpf.make_params(storage, **p)] * 2)
    alone = lbpf.Sim(shape, lattices, storage=storage, **p)
    _init([batch.sims[0], alone])
    _init([batch.sims[1]])
    batch.step(13)
    alone.step(13)
    _same(batch.sims[0], alone, state=True)
    batch.close()


# D2Q9 phi as planes in BF16, and narrow rows: phi tiled beside planes, node-wise beyond the lines of wide rows
@pytest.mark.parametrize("storage,shape,lattices", [("bf16", (1030, 1100, 1), (9, 5, 5)), ("f32", (120, 36700, 1), (9, 9, 9)),
                                                    ("f32", (24, 200000, 1), (9, 5, 5)), ("f32", (64, 15625, 1), (9, 9, 0)),
                                                    ("f16", (31, 22580, 1), (5, 9, 5))])
def test_narrow_forms_equal_tiles(storage, shape, lattices):
    p = workloads.base_params(kappa=100.0)
    shapes = [shape, (1101, 1100, 1)]
    batch = lbpf.Batch.create(shapes, lattices, [lbpf.make_params(storage, **p) for _ in shapes])
    alone = lbpf.Sim(shape, lattices, storage=storage, **p)
    _init([batch.sims[0], alone])
    _init([batch.sims[1]])
    batch.step(7)
    alone.step(7)
    _same(batch.sims[0], alone, state=True)
    batch.close()
