"""The node-wise step (collisions without a halo, moments in a pass of their own) where it can
go wrong: against the oracle at a size where a block spans several planes, and bit for bit
against the tiled step where a batch and its members take different forms."""
import numpy as np
import pytest

import oracle
from paper_1602_07483_gb300 import lbpf, workloads

pytestmark = pytest.mark.gpu


def _pair(shape, lattices, seed=3):
    p = workloads.base_params(kappa=100.0)
    centres = np.array([[s // 2 if s > 1 else 0 for s in shape]], np.float64)
    radii = np.array([6.0])
    ora = oracle.Sim(shape, lattices, params=oracle.make_params(**p))
    ora.init_seed(centres, radii, -0.55, -0.3)
    noise = workloads.population_noise(shape, lattices, seed=seed)
    state = [None if n is None else ora.pops(f) + n for f, n in enumerate(noise)]
    ora.set_state(*state, theta0=-0.3)
    gpu = lbpf.Sim(shape, lattices, storage="f64", **p)
    gpu.set_state(*state, theta0=-0.3)
    return gpu, ora


# rows and planes that are no multiple of a block, blocks of two and of three planes with a
# ragged last one, a plane smaller than a block; one step from the same noisy state: the
# bound of the other one-step parity tests (1e-12 of the largest value)
@pytest.mark.parametrize("shape,lattices", [((101, 104, 99), (19, 19, 7)), ((127, 130, 101), (15, 7, 0)),
                                            ((11, 10, 61), (7, 15, 19))])
def test_blocks_of_several_planes_match_oracle(shape, lattices):
    gpu, ora = _pair(shape, lattices)
    gpu.step(1)
    ora.step(1)
    for a, b in zip(gpu.read_fields(), ora.fields()):
        assert np.abs(a - b).max() <= 1e-12 * max(1.0, np.abs(b).max())
    for f, a in enumerate(gpu.get_state()):
        if a is not None:
            b = ora.pops(f)
            assert np.abs(a - b).max() <= 1e-12 * max(1.0, np.abs(b).max())


# a batch large enough to run tiled over members that run node-wise alone: the same values
@pytest.mark.parametrize("shapes,lattices", [([(151, 149, 150)] * 3, (19, 19, 19)), ([(701, 500, 1), (640, 700, 1)], (9, 5, 9))])
def test_tiled_batch_equals_node_wise_members(shapes, lattices):
    p = dict(workloads.base_params(kappa=100.0), aniso=1, eps1=-0.02, eps2=0.015, dt=0.01)
    batch = lbpf.Batch.create(shapes, lattices, [lbpf.make_params("f32", **p) for _ in shapes])
    alone = [lbpf.Sim(s, lattices, storage="f32", **p) for s in shapes]
    for k, (a, b) in enumerate(zip(batch.sims, alone)):
        c = np.array([[20.0 + k, 15.0, 0.0 if shapes[k][2] == 1 else 9.0]])
        for s in (a, b):
            s.init_seed(c, np.array([7.0]), -0.5, -0.3)
    batch.step(8)
    for a, b in zip(batch.sims, alone):
        b.step(8)
        for x, y in zip(a.read_fields(), b.read_fields()):
            assert np.array_equal(x, y)
    batch.close()


# rows of even length step two nodes per thread; in a batch with one odd row length every member
# takes one node per thread: the same values.  Rows shorter and longer than a warp's span, one and
# two pairs long, thin boxes, D3Q7 to D3Q19, and both 2D lattices.
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("shapes,lattices", [([(48, 20, 18), (2, 9, 7), (66, 5, 3), (33, 12, 10)], (19, 19, 19)),
                                             ([(4, 31, 6), (130, 7, 9), (31, 12, 10)], (15, 7, 15)),
                                             ([(40, 1, 5), (62, 17, 16), (25, 12, 10)], (7, 15, 0)),
                                             ([(258, 40, 1), (2, 77, 1), (91, 33, 1)], (9, 9, 5)),
                                             ([(64, 50, 1), (91, 33, 1)], (5, 5, 9))])
def test_pairs_equal_single_nodes(storage, shapes, lattices):
    p = dict(workloads.base_params(kappa=100.0))
    batch = lbpf.Batch.create(shapes, lattices, [lbpf.make_params(storage, **p) for _ in shapes])
    alone = [lbpf.Sim(s, lattices, storage=storage, **p) for s in shapes]
    for k, (a, b) in enumerate(zip(batch.sims, alone)):
        c = np.array([[0.4 * shapes[k][0], 0.6 * shapes[k][1], 0.4 * (shapes[k][2] - 1)]])
        for s in (a, b):
            s.init_seed(c, np.array([4.0]), -0.55, -0.3)
    batch.step(13)
    for a, b in zip(batch.sims, alone):
        b.step(13)
        for x, y in zip(a.read_fields(), b.read_fields()):
            assert np.isfinite(x).all() and np.array_equal(x, y)
        for x, y in zip(a.get_state(), b.get_state()):
            assert x is None or np.array_equal(x, y)
    batch.close()


# planes large enough for the warp-per-tile step (rows of even length), whole and ragged last tiles,
# one chunk and many; in a batch with one odd row length every member runs the tiled form of one
# node per thread: the same values
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("shape,lattices", [((1020, 1300, 1), (9, 5, 5)), ((1262, 1001, 1), (5, 9, 9)),
                                            ((32, 40000, 1), (9, 9, 0)), ((3202, 3800, 1), (9, 5, 9)), ((150002, 9, 1), (9, 9, 5)),
                                            ((1400002, 1, 1), (5, 5, 9))])
def test_planes_equal_single_nodes(storage, shape, lattices):
    p = dict(workloads.base_params(kappa=100.0))
    shapes = [shape, (901, 900, 1)]
    batch = lbpf.Batch.create(shapes, lattices, [lbpf.make_params(storage, **p) for _ in shapes])
    alone = lbpf.Sim(shape, lattices, storage=storage, **p)
    c = np.array([[0.0, 0.0, 0.0], [0.7 * shape[0], 0.6 * shape[1], 0.0]])
    for s in (batch.sims[0], alone):
        s.init_seed(c, np.array([9.0, 12.0]), -0.55, -0.3)
    batch.sims[1].init_seed(c[:1], np.array([9.0]), -0.55, -0.3)
    batch.step(7)
    alone.step(7)
    for x, y in zip(batch.sims[0].read_fields(), alone.read_fields()):
        assert np.isfinite(x).all() and np.array_equal(x, y)
    batch.close()
