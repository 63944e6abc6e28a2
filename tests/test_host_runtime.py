"""The host side of the library (work lists, graphs, uploads) without a GPU.

The compiled objects are linked against tests/fake_cudart.cpp in place of the CUDA runtime: every
launch of a step kernel is checked to read live memory whose upload is ordered before it, and
recorded, and allocations can be made to fail.
"""
import ctypes
import os
import subprocess

import pytest

from paper_1602_07483_gb300 import build, lbpf

HERE = os.path.dirname(os.path.abspath(__file__))


class Fake:
    def __init__(self, lib):
        self.lib = lib
        lib.fake_launch.restype = lib.fake_violation.restype = ctypes.c_char_p

    def clear(self):
        self.lib.fake_clear()

    def fail_malloc(self, after, count=1):
        self.lib.fake_fail_malloc(after, count)

    def violations(self):
        return [self.lib.fake_violation(i).decode() for i in range(self.lib.fake_violations())]

    def launches(self):
        """(kernel, blocks, threads, planes of the first and of the longest work item)"""
        return [self.lib.fake_launch(i).decode() for i in range(self.lib.fake_launches())]


@pytest.fixture(scope="module")
def fake_path(tmp_path_factory):
    build.build()
    out = str(tmp_path_factory.mktemp("fake") / "liblbpf_fake.so")
    objs = [os.path.join(build.OUT_DIR, "obj", s.replace(".cu", ".o")) for s in build.SOURCES]
    subprocess.run([build.nvcc(), "-std=c++17", "-shared", "-cudart", "none", "-Xcompiler", "-fPIC,-Wall", "-Xlinker",
                    "-Bsymbolic", "-o", out, os.path.join(HERE, "fake_cudart.cpp")] + objs, check=True)
    return out


@pytest.fixture
def fake(fake_path, monkeypatch):
    monkeypatch.setattr(lbpf, "_LIB", None)
    f = Fake(lbpf.load(fake_path))
    f.fail_malloc(-1, 0)
    f.clear()
    yield f
    f.fail_malloc(-1, 0)


# 3D and 2D, node-wise, tiled and plane forms, and mixed ones
SIMS = [((32, 32, 32), (15, 19, 0), "f64"), ((33, 20, 18), (19, 19, 7), "f32"), ((202, 202, 202), (19, 19, 19), "f32"),
        ((64, 48, 1), (9, 5, 5), "f16"), ((1200, 1000, 1), (9, 5, 5), "f32"), ((1600, 1500, 1), (9, 5, 5), "bf16")]


@pytest.mark.parametrize("shape,lattices,storage", SIMS)
@pytest.mark.parametrize("schedule", ["two_kernels", "one_launch"])
def test_uploads_are_ordered_before_the_steps(fake, shape, lattices, storage, schedule):
    s = lbpf.Sim(shape, lattices, storage=storage)
    if schedule == "one_launch":
        try:
            s.set_schedule(schedule)
        except lbpf.LbpfError:
            pytest.skip("no one-launch step for these lattices and storage")
    s.step(7)
    s.set_tiling(4, 5)
    s.step(7)
    b = lbpf.Batch([s])
    b.step(7)
    b.set_tiling(6, 4)
    b.step(7)
    assert len(fake.launches()) >= 28
    assert fake.violations() == []
    b.close()


@pytest.mark.parametrize("shape,lattices,storage", SIMS)
@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("schedule", ["two_kernels", "one_launch"])
def test_a_failed_tiling_keeps_the_old_one(fake, shape, lattices, storage, batched, schedule):
    """Whichever allocation fails, the call reports it and the steps run on as planned before."""
    s = lbpf.Sim(shape, lattices, storage=storage)
    s = lbpf.Batch([s]) if batched else s
    if schedule == "one_launch":
        try:
            s.set_schedule(schedule)
        except lbpf.LbpfError:
            pytest.skip("no one-launch step for these lattices and storage")

    def steps():
        fake.clear()
        s.step(6)  # a graph
        s.step(5)
        s.step(1)
        assert fake.violations() == []
        return fake.launches()

    def fails(call):
        """Runs the call with its first, second, ... allocation failing until it succeeds."""
        for after in range(20):
            fake.fail_malloc(after)
            try:
                call()
            except lbpf.LbpfError as e:
                if e.code == lbpf.LBPF_EINVAL:  # no one-launch step for these lattices and storage
                    return 2
                assert e.code == lbpf.LBPF_ENOMEM
            else:
                fake.fail_malloc(-1, 0)
                return after
            fake.fail_malloc(-1, 0)
            assert steps() == before
            assert s.schedule == schedule
            if not batched:
                assert s.get_tiling() == tiling
        raise AssertionError("never succeeded")

    before, tiling = steps(), s.get_tiling()
    assert fails(lambda: s.set_tiling(4, 5)) >= 2
    before, tiling = steps(), s.get_tiling()
    assert fails(lambda: s.set_schedule("one_launch" if schedule == "two_kernels" else "two_kernels")) >= 2
    fake.fail_malloc(-1, 0)
    steps()
    s.close()


@pytest.mark.parametrize("shape,lattices,storage", SIMS)
def test_tuning_starts_from_the_tiling_in_use(fake, shape, lattices, storage):
    """Setting the reported tiling changes nothing, and tuning never ends slower than it began:
    phi of the 202^3 box runs node-wise and U and theta tiled, with chunks of their own."""
    s = lbpf.Sim(shape, lattices, storage=storage)

    def step():
        fake.clear()
        ms = s.step_timed(6)[2]
        return fake.launches(), ms

    launches, ms = step()
    s.set_tiling(*((0, s.get_tiling()[1]) if shape[2] == 1 else s.get_tiling()))
    assert step() == (launches, ms)
    s.set_tiling(8, 0)
    before, ms = step()
    assert before == launches
    s.autotune(6)
    assert step()[1] <= ms
    s.set_tiling(8, 1000)
    assert s.get_tiling()[1] == 1000
    s.set_schedule("two_kernels")
    assert s.get_tiling()[1] == 1000


@pytest.mark.parametrize("shape,lattices,storage", SIMS)
def test_step_launches_counts_the_kernels(fake, shape, lattices, storage):
    s = lbpf.Sim(shape, lattices, storage=storage)
    for schedule in ("two_kernels", "one_launch"):
        try:
            s.set_schedule(schedule)
        except lbpf.LbpfError:
            continue
        fake.clear()
        s.step(8)
        assert len(fake.launches()) == 8 * s.step_launches


# the form of each phase on both sides of the lines that choose it: narrow rows count with their idle
# lanes, 16 bits and FP32 and odd rows have lines of their own, U and theta theirs
NODE, PAIR, TILE, PLANE = ("node", "moment"), ("pair", "moment2"), ("",), ("plane",)
FORMS = [((500, 500, 1), (9, 5, 5), "f32", PAIR, PAIR), ((900, 900, 1), (9, 5, 5), "f32", TILE, PLANE),
         ((900, 900, 1), (9, 9, 9), "f32", TILE, TILE), ((100000, 8, 1), (9, 5, 5), "f32", TILE, PLANE),
         ((16, 60000, 1), (9, 5, 5), "f32", TILE, PLANE), ((16, 8000, 1), (9, 5, 5), "f32", PAIR, PAIR),
         ((2200, 2200, 1), (9, 9, 9), "f32", PLANE, PLANE), ((841, 841, 1), (9, 5, 5), "f32", TILE, TILE),
         ((701, 701, 1), (9, 5, 5), "f32", NODE, NODE), ((1000, 1000, 1), (9, 9, 9), "f16", PAIR, PAIR),
         ((1100, 1100, 1), (9, 9, 9), "bf16", PLANE, PLANE), ((1001, 1001, 1), (9, 5, 5), "f16", NODE, NODE),
         ((1301, 1301, 1), (9, 5, 5), "f16", TILE, TILE), ((3000, 3000, 1), (9, 5, 5), "f64", NODE, NODE),
         ((202, 202, 202), (19, 15, 15), "f32", PAIR, TILE), ((203, 203, 203), (19, 15, 15), "f32", TILE, TILE),
         ((203, 203, 203), (19, 19, 7), "f32", NODE, NODE), ((203, 203, 203), (19, 19, 19), "bf16", NODE, NODE)]


@pytest.mark.parametrize("shape,lattices,storage,phi,uth", FORMS)
def test_forms(fake, shape, lattices, storage, phi, uth):
    s = lbpf.Sim(shape, lattices, storage=storage)
    s.step(1)
    names = [l.split()[0] for l in fake.launches()]
    want = [("k_phi_" if k else "k_phi") + k for k in phi] + [("k_uth_" if k else "k_uth") + k for k in uth]
    assert len(names) == len(want)
    for n, w in zip(names, want):
        assert "%d%sI" % (len(w), w) in n


def test_narrow_rows_take_whole_warps(fake):
    for shape, threads in (((40, 400, 1), 32), ((90, 200, 1), 64), ((256, 20, 1), 128), ((300, 20, 1), 128)):
        s = lbpf.Sim(shape, (9, 5, 5), storage="f32")
        fake.clear()
        s.step(1)
        assert {int(l.split()[2]) for l in fake.launches()} == {threads}


def test_plane_chunks_fill_whole_waves(fake):
    """One-warp blocks, 24 to an SM: one wave where chunks of 8 to 48 rows make one, else 32 rows."""
    for shape in ((2000, 2000, 1), (2100, 2100, 1), (3000, 3000, 1), (1030, 1100, 1)):
        s = lbpf.Sim(shape, (9, 5, 5), storage="f16")
        fake.clear()
        s.step(1)
        for l in fake.launches():
            name, blocks, _, _, rows = l.split()
            assert "plane" in name and 8 <= int(rows) <= 48 and int(blocks) <= 152 * 24
            assert int(blocks) > 0.9 * 152 * 24 or int(rows) == 8
    s = lbpf.Sim((5000, 5000, 1), (9, 5, 5), storage="f16")
    fake.clear()
    s.step(1)
    assert [l.split()[-1] for l in fake.launches()] == ["32", "32"]


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
def test_every_pairing_has_its_kernels(fake, storage):
    """Tiled kernels exist only where some size takes them: every pairing steps, on both sides of the lines."""
    for shape, qs in (((203, 203, 203), (7, 15, 19)), ((24, 20, 16), (7, 15, 19)), ((1301, 1301, 1), (5, 9)),
                      ((2200, 2200, 1), (5, 9)), ((900, 900, 1), (5, 9)), ((40, 30, 1), (5, 9))):
        for qu in qs:
            for qt in qs + (0,):
                s = lbpf.Sim(shape, (qs[0], qu, qt), storage=storage)
                s.step(1)
                s.set_tiling(5, 0)
                s.step(1)
                s.close()
    assert fake.violations() == []


def test_blocks_of_small_planes_stay_whole_where_few_of_them_run(fake):
    """FP64 and 3D: whole blocks until there are more of them than the chip holds; in a batch all members count."""
    for shapes, lattices, storage, threads in (
            ([(64, 500, 1)], (9, 5, 5), "f64", 128), ([(64, 2999, 1)], (9, 5, 5), "f64", 128), ([(24, 3000, 1)], (9, 5, 5), "f64", 32),
            ([(4, 4, 800)], (19, 19, 7), "f64", 128), ([(6, 16, 1999)], (19, 19, 7), "f32", 128),
            ([(6, 16, 2000)], (19, 19, 7), "f32", 64), ([(6, 16, 1000)] * 2, (19, 19, 7), "f32", 64),
            ([(12, 12, 300)], (19, 19, 7), "f16", 128), ([(12, 12, 1200)], (19, 19, 7), "bf16", 96)):
        b = lbpf.Batch([lbpf.Sim(s, lattices, storage=storage) for s in shapes])
        fake.clear()
        b.step(1)
        assert {int(l.split()[2]) for l in fake.launches()} == {threads}, (shapes, storage)
        b.close()


# narrow rows beyond the lines of wide ones: node-wise where tiles or planes idle more lanes than node-wise blocks
NARROW_FORMS = [((31, 22580, 1), (9, 5, 5), "f32", NODE, NODE), ((45, 33333, 1), (9, 9, 9), "bf16", NODE, NODE),
                ((91, 60000, 1), (9, 5, 5), "f16", TILE, TILE), ((64, 15625, 1), (9, 9, 9), "f32", PAIR, PAIR),
                ((128, 11718, 1), (5, 5, 0), "f16", PAIR, PAIR), ((128, 40000, 1), (9, 5, 5), "f32", PLANE, PLANE),
                ((48, 20834, 1), (9, 5, 5), "f32", TILE, PLANE), ((160, 12500, 1), (9, 5, 5), "f16", PLANE, PLANE),
                ((97, 5154, 1), (9, 5, 5), "f32", NODE, NODE), ((97, 7216, 1), (9, 5, 5), "f32", TILE, TILE),
                ((300, 1666, 1), (5, 5, 0), "f32", PAIR, PAIR), ((300, 2333, 1), (9, 9, 9), "f16", PAIR, PAIR),
                ((300, 2333, 1), (9, 5, 5), "f16", PLANE, PLANE), ((48, 83333, 1), (9, 9, 9), "f32", PLANE, PLANE),
                ((24, 291666, 1), (9, 9, 9), "f32", TILE, PLANE), ((24, 180000, 1), (9, 9, 9), "f32", TILE, TILE),
                ((201, 3980, 1), (5, 5, 0), "f16", TILE, TILE), ((201, 3400, 1), (5, 5, 0), "f16", NODE, NODE),
                ((1000, 800, 1), (5, 5, 0), "f32", PAIR, PAIR), ((1000, 800, 1), (9, 5, 5), "f32", TILE, PLANE),
                ((45, 66666, 1), (9, 9, 9), "f32", TILE, TILE), ((91, 16483, 1), (9, 5, 5), "f32", NODE, NODE),
                ((120, 35833, 1), (9, 9, 9), "f32", TILE, PLANE), ((97, 6701, 1), (9, 9, 0), "f32", NODE, NODE),
                ((15, 60000, 1), (5, 9, 9), "f32", TILE, TILE), ((1000, 800, 1), (5, 9, 9), "f32", PAIR, PAIR)]


@pytest.mark.parametrize("shape,lattices,storage,phi,uth", NARROW_FORMS)
def test_forms_of_narrow_rows(fake, shape, lattices, storage, phi, uth):
    test_forms(fake, shape, lattices, storage, phi, uth)
