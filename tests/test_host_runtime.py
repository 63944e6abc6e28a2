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
            if "plane" not in name:
                continue
            assert 8 <= int(rows) <= 48 and int(blocks) <= 152 * 24
            assert int(blocks) > 0.9 * 152 * 24 or int(rows) == 8
    s = lbpf.Sim((5000, 5000, 1), (9, 5, 5), storage="f16")
    fake.clear()
    s.step(1)
    assert {l.split()[-1] for l in fake.launches() if "plane" in l} == {"32"}
