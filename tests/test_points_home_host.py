"""The host side's choice of where a world's points live, on a device made of host memory: two SMs
that hold three blocks with the points in shared memory and eight with them in global memory."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2411_05799_gb300 import build, npx, scenes

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    include = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", include, "-o", out,
                    os.path.join(HERE, "fake_device.cpp"), os.path.join(build.CSRC, "npx_world.cpp")], check=True)
    lib = C.CDLL(out)
    for name, args in npx._SIGS.items():
        if hasattr(lib, name):
            getattr(lib, name).argtypes = args
            getattr(lib, name).restype = C.c_int
    lib.npx_last_error.restype = C.c_char_p
    lib.fake_fail_bytes.argtypes = [C.c_size_t]
    lib.fake_launches.argtypes = [C.c_void_p, C.c_int]
    return lib


@pytest.fixture
def dev(fake, monkeypatch):
    monkeypatch.setattr(npx, "_lib", fake)
    yield fake
    fake.fake_fail_bytes(0)


def _bodies(count, points, K=80):
    return scenes.ragged_bodies([points] * count).with_(joint_update_steps=K)


def _world(b, lanes=8, warps=2):
    w = npx.World.from_batch(b, configure=dict(lanes_per_scene=lanes, warps_per_block=warps))
    w.use_graphs(False)
    return w


def _launches(dev, w, n):
    dev.fake_clear()
    w.step(n)
    a = np.zeros((64, 6), np.int64)
    return a[:dev.fake_launches(a.ctypes.data, 64)]


# 8 lanes, 2 warps: 8 scenes a block, 48 at once in the slots, 128 in global memory
@pytest.mark.parametrize("robots, points, K, steps, gp", [
    (48, 200, 80, 100, 0),                                            # all fit in the slots
    (49, 200, 80, 1, 1), (128, 200, 20, 1, 1), (128, 200, 19, 1, 0),  # all fit in global memory
    (129, 200, 40, 16, 1), (129, 200, 40, 15, 0), (129, 200, 39, 16, 0), (166, 200, 40, 15, 0),   # a short tail
    (167, 200, 20, 1, 1)])                                            # a long one
def test_the_rule(dev, robots, points, K, steps, gp):
    w = _world(_bodies(robots, points, K))
    (l,) = _launches(dev, w, steps)
    assert l[0] == gp and l[1] == steps
    if gp:
        assert l[4] >= l[2] * l[3] * 4 * points   # the launch's scenes in flight have room
    w.close()


def test_scenes_of_many_points(dev):
    w = _world(_bodies(100, 600), lanes=16)
    assert [_launches(dev, w, n)[0][0] for n in (15, 16)] == [0, 1]
    w.close()


def test_a_remainder_of_few_steps_stays_in_the_slots(dev):
    w = _world(_bodies(140, 200))
    w.configure(chunk_steps=20)
    assert [tuple(l[:2]) for l in _launches(dev, w, 45)] == [(1, 20), (1, 20), (0, 5)]
    w.close()


def test_without_memory_the_points_stay_in_the_slots(dev):
    """The scratch's allocation fails: the world steps all the same, here and after changes that would
    lay it out again."""
    points = 200
    dev.fake_fail_bytes(16 * 16 * 8 * points)   # 16 blocks of 8 scenes, one more than there are
    w = _world(_bodies(127, points))
    (l,) = _launches(dev, w, 50)
    assert tuple(l[:3]) == (0, 50, 6)
    w.set_friction_model(3)
    w.set_friction_model(0)
    assert _launches(dev, w, 50)[0][0] == 0
    w.configure(lanes_per_scene=8, warps_per_block=1)
    assert tuple(_launches(dev, w, 50)[0][:4]) == (0, 50, 6, 1)
    w.close()


def test_size_classes_do_not_share_their_scratch(dev):
    b = scenes.ragged_bodies([100] * 300 + [400] * 300)
    w = npx.World.from_batch(b)
    w.use_graphs(False)
    ls = _launches(dev, w, 50)
    assert len(ls) == 2 and (ls[:, 0] == 1).all()
    spans = sorted((l[5], l[5] + l[2] * l[3] * 2 * p) for l, p in zip(ls, (400, 100)))
    assert spans[0][1] <= spans[1][0] and (ls[:, 4] >= [ls[0][2] * ls[0][3] * 2 * 400, ls[1][2] * ls[1][3] * 2 * 100]).all()
    w.close()
