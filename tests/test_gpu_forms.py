"""Node-wise blocks of fewer warps, bit for bit against whole ones."""
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
