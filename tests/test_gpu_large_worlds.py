"""Worlds of more scenes than fit on the device at once keep the posed points of the scenes in flight
in global memory (an explicit grid keeps them in shared memory); shapes at the edge of shared memory."""
import numpy as np
import pytest

from paper_2411_05799_gb300 import scenes
from paper_2411_05799_gb300.npx import NpxError, World

pytestmark = pytest.mark.gpu

KEYS = ("cog", "quat", "vel", "omega", "angmom", "theta", "contacts", "status")


def _after(b, steps, programs=None, **shape):
    w = World.from_batch(b, configure=shape or None)
    if programs is not None:
        w.set_gp_programs(programs)
    for n in steps:
        w.step(n)
    r = w.read()
    r["kappa"] = w.contacts()
    w.close()
    return r


@pytest.mark.parametrize("batch, lanes, warps", [
    ("hexapods", 8, 2), ("hexapods", 16, 3), ("hexapods", 32, 1), ("quadrupeds", 4, 2), ("uneven", 16, 4),
    ("bodies", 8, 4), ("controllers", 8, 2)])
def test_points_in_global_memory_change_nothing(batch, lanes, warps):
    """Same lanes, same arithmetic: bit for bit what the explicit grid of one block per SM gives, over
    joint updates, in chunks of uneven lengths, and for point counts that leave tiles part full."""
    progs = None
    if batch == "hexapods":
        b = scenes.hexapod_batch(9001, seed_key=3)
    elif batch == "controllers":
        b = scenes.hexapod_batch(8000, seed_key=3)
        progs = np.random.default_rng(1).integers(0, 256, (8000, 32), dtype=np.uint8)
    elif batch == "quadrupeds":
        b = scenes.legged_batch(20001, 4, seed_key=3)
    elif batch == "bodies":
        b = scenes.ragged_bodies([1 + (37 * i) % 512 for i in range(30000)], seed_key=3)
    else:
        b = scenes.uneven_batch(6000, seed_key=3)
    steps = (1, 85, 160)
    free = dict(lanes_per_scene=lanes, warps_per_block=warps)
    r = _after(b, steps, progs, **({} if batch == "uneven" else free))
    ref = _after(b, steps, progs, **free, blocks=152)
    for k in KEYS + ("kappa",):
        np.testing.assert_array_equal(r[k], ref[k], err_msg=k)
    assert (r["status"] == 0).mean() > 0.99


def test_shapes_at_the_edge_of_shared_memory():
    """A shape whose slots fill shared memory but for the links' tree numbers is taken (with fewer warps
    per block), one that never fitted is refused; the results are those of any other shape."""
    # 64 links and 876 points at 16 lanes: 12 slots of 19,360 bytes are 232,320 of a block's 232,448
    pts = np.random.default_rng(0).uniform(-0.1, 0.1, (876, 3)).astype(np.float32)
    n = np.full(64, 13)
    n[:44] += 1
    off = np.concatenate([[0], np.cumsum(n)])
    links = [((0.2, 0.2, 0.2), (0, 0, 0), 1.0, k - 1, (0.0, 0.0, 0.0) if k else None,
              (0.0, 0.0, 1.0) if k else None, -1) for k in range(64)]
    b = scenes._assemble([(links, [pts[off[k]:off[k + 1]] for k in range(64)])] * 20, mu=np.full(20, 0.6),
                         origin=np.tile([0, 0, 0.3], (20, 1)), quat=np.tile([1.0, 0, 0, 0], (20, 1)),
                         vel=np.zeros((20, 3)), omega=np.tile([0.3, 0.2, 0.1], (20, 1)), act_params=None,
                         name="edge", act_mode=scenes.ACT_HOLD)
    fits = 6
    r = _after(b, (50,), lanes_per_scene=16, warps_per_block=fits)
    ref = _after(b, (50,), lanes_per_scene=16, warps_per_block=2)
    for k in KEYS:
        np.testing.assert_array_equal(r[k], ref[k], err_msg=k)
    with pytest.raises(NpxError):
        _after(b, (1,), lanes_per_scene=16, warps_per_block=fits + 1)


def test_autotuned_shapes_agree():
    """The autotuner times both homes of the points; what it settles on gives the bits of an explicit
    grid with the same lanes."""
    b = scenes.hexapod_batch(9001, seed_key=5)
    w = World.from_batch(b)
    lanes = w.autotune(20)["lanes_per_scene"]
    ref = World.from_batch(b, configure=dict(lanes_per_scene=lanes, warps_per_block=1, blocks=152))
    for x in (w, ref):
        x.step(200)
    r, q = w.read(), ref.read()
    for k in KEYS:
        np.testing.assert_array_equal(r[k], q[k], err_msg=k)
    w.close()
    ref.close()
