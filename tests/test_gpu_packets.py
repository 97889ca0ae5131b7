"""The packet phase (a warp's rays walk the tree together) returns what the
per-ray traversal returns, bit for bit: the casts with default options against
the same casts with lane-serial leaf tests (tri_mode 1), which never use
packets.  Over sensors whose packets are narrow, wide, partial or shorter than
half a warp, environments whose ray count is no multiple of 32, both widths,
minimum ranges, poses looking along every axis, leaning, scaled, far outside
the scene, on the scene's own planes and not finite, packets of 32 and 96 rays
and blocks without room for the packet lists."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


def scene_parts(kind):
    if kind == "boxes":
        v, t, _ = synth.tiny_room_scene(3)
        return v, t, np.array([10.0, 8.0, 3.0])
    v, t, _ = synth.indoor_scene(5, n_spheres=120, n_boxes=60)
    return v, t, np.array([20.0, 15.0, 4.0])


def poses(room, n=24):
    rng = np.random.default_rng(11)
    p = synth.random_rotation(rng, n) if hasattr(synth, "random_rotation") else None
    if p is None:
        from synth.poses import random_rotation
        p = random_rotation(rng, n)
    pos = 0.05 + rng.uniform(0, 1, (n, 3)) * (room - 0.1)
    # along the axes, exactly
    axes = [np.eye(3), np.diag([-1.0, -1, 1]), np.array([[0.0, -1, 0], [1, 0, 0], [0, 0, 1]]),
            np.array([[0.0, 0, 1], [0, 1, 0], [-1, 0, 0]]), np.array([[0.0, 0, -1], [0, 1, 0], [1, 0, 0]])]
    for k, a in enumerate(axes):
        p[k] = a
    pos[5] = room * 40.0                               # far outside
    pos[6] = [-30.0, room[1] / 2, room[2] / 2]
    pos[7] = [0.0, 0.0, 0.0]                           # a corner of the room
    pos[8] = [room[0] / 2, 0.0, room[2] / 2]           # on a wall
    p[9] *= 2.5                                        # rays not of unit length
    p[10] *= 1e-3
    P = np.concatenate([p, pos[:, :, None]], 2).astype(np.float32)
    P[11, 0, 0] = np.nan
    P[12, 1, 3] = np.inf
    P[13, :, :3] = 0.0                                 # rays without a direction
    return P


def sensors():
    g = synth.grid_sensor
    dense = g(32, -1.0, 1.0, 64)
    return {"16x360": (g(16, -15, 15, 360), {}), "dense": (dense, {}), "7x45": (g(7, -30, 30, 45), {}),
            "5x7": (g(5, -10, 10, 7), {}), "one": (g(1, 0, 0, 1), {}), "up": (g(24, 60, 90, 48), {}),
            "rosette": (synth.rosette_sensor(1000, 2), {}), "rows": (g(16, -15, 15, 100), dict(tile_rows=1, tile_cols=32))}


def cast(item, opts):
    sc, se, P, far, near = item
    n = len(P) * se.n_rays
    r = torch.full((n,), -7.0, dtype=torch.float32, device="cuda")
    i = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    fgl.cast_batched([(sc, se, P, far, r, i, near)], opts)
    fgl.sync()
    return r, i


@pytest.mark.parametrize("kind", ["boxes", "indoor"])
@pytest.mark.parametrize("width", [8, 4])
@pytest.mark.parametrize("name", list(sensors()))
def test_packets_equal_per_ray_casts(kind, width, name):
    v, t, room = scene_parts(kind)
    sc = fgl.Scene(v, t, width=width)
    tab, kw = sensors()[name]
    se = fgl.Sensor.from_table(tab, **kw)
    P = torch.from_numpy(poses(room)).cuda()
    for far, near in ((100.0, 0.0), (3.0, 0.0), (30.0, 0.7)):
        item = (sc, se, P, far, near)
        ref = cast(item, fgl.BatchOpts(tri_mode=1))
        for opts in (None, fgl.BatchOpts(packet_rays=96), fgl.BatchOpts(block_threads=256, stack_smem=2),
                     fgl.BatchOpts(block_threads=448, stack_smem=21), fgl.BatchOpts(refill_min=8)):
            got = cast(item, opts)
            assert torch.equal(ref[0].view(torch.int32), got[0].view(torch.int32)) and torch.equal(ref[1], got[1])
        if near == 0.0:
            n = len(P) * se.n_rays
            for opts in (fgl.BatchOpts(), fgl.BatchOpts(block_threads=64, stack_smem=1), fgl.BatchOpts(count_work=1)):
                r, i = fgl.cast_opts(sc, se, P, far, opts)
                fgl.sync()
                assert torch.equal(ref[0].view(torch.int32), r.view(torch.int32)) and torch.equal(ref[1], i)
            r, i = fgl.cast(sc, se, P, far)
            fgl.sync()
            assert r.numel() == n
            assert torch.equal(ref[0].view(torch.int32), r.view(torch.int32)) and torch.equal(ref[1], i)


def test_mixed_batch_and_static_form():
    """Narrow and wide sensors, both widths and a minimum range in one batch
    (the groups' kernels follow the majority), also through the form without
    allocations."""
    v, t, room = scene_parts("indoor")
    scenes = [fgl.Scene(v, t, width=w) for w in (8, 4)]
    tabs = sensors()
    P = torch.from_numpy(poses(room)).cuda()
    for names in (("16x360", "rosette", "5x7", "dense"), ("rosette", "one", "5x7"), ("7x45", "rosette")):
        outs = {}
        for mode in ("serial", "default", "static"):
            items = []
            for k, nm in enumerate(names):
                se = fgl.Sensor.from_table(tabs[nm][0])
                n = len(P) * se.n_rays
                items.append((scenes[k % 2], se, P, 50.0, torch.empty(n, device="cuda"),
                              torch.empty(n, dtype=torch.int32, device="cuda"), 0.4 if k == 1 else 0.0))
            if mode == "static":
                fgl.cast_batched_static(items)
            else:
                fgl.cast_batched(items, fgl.BatchOpts(tri_mode=1) if mode == "serial" else None)
            fgl.sync()
            outs[mode] = [(x[4], x[5]) for x in items]
        for mode in ("default", "static"):
            for (r0, i0), (r1, i1) in zip(outs["serial"], outs[mode]):
                assert torch.equal(r0.view(torch.int32), r1.view(torch.int32)) and torch.equal(i0, i1)


# either side of the size up to which a packet is 16 rays (136,192 rays), whole
# and partial packets: one launch, the batch and the batch without allocation
@pytest.mark.parametrize("beams,az,envs", [(16, 266, 32), (16, 267, 32), (7, 45, 432), (7, 45, 433), (5, 9, 1)])
def test_small_and_large_casts(beams, az, envs):
    v, t, room = scene_parts("boxes")
    sc = fgl.Scene(v, t)
    se = fgl.Sensor.from_table(synth.grid_sensor(beams, -20, 20, az))
    P = torch.from_numpy(np.resize(poses(room), (envs, 3, 4))).cuda()
    ref = cast((sc, se, P, 50.0, 0.0), fgl.BatchOpts(tri_mode=1))
    got = [cast((sc, se, P, 50.0, 0.0), None), cast((sc, se, P, 50.0, 0.0), fgl.BatchOpts(packet_rays=32)),
           fgl.cast(sc, se, P, 50.0)]
    r, i = torch.empty_like(ref[0]), torch.empty_like(ref[1])
    fgl.cast_batched_static([(sc, se, P, 50.0, r, i)])
    fgl.sync()
    for a, b in got + [(r, i)]:
        assert torch.equal(a.reshape(-1).view(torch.int32), ref[0].view(torch.int32)) and torch.equal(b.reshape(-1), ref[1])
