"""Which casts walk packets of rays together: the sizes on either side of each
line of the rule -- sensors of few rays and of half-empty packets, coarse and fine
ones, scenes of 108 to 64,000 triangles, nearly empty and cluttered, and of 5,000 to
4,300,000 rays -- return what the lane-serial form returns, bit for bit, over the host-built
tree, alone, in a batch and without allocations, and over the GPU-built one."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


def field(rows, cols):
    """rows x cols rays over 20 x 20 degrees."""
    el, az = np.deg2rad(np.linspace(-10, 10, rows)), np.deg2rad(np.linspace(-10, 10, cols))
    E, A = np.meshgrid(el, az, indexing="ij")
    return fgl.Sensor(E.reshape(-1).astype(np.float32), A.reshape(-1).astype(np.float32), rows, cols)


def sensor(name):
    if name.startswith("field"):
        return field(*map(int, name[5:].split("x")))
    return fgl.Sensor.from_table(synth.grid_sensor(*{"16x360": (16, -15, 15, 360), "5x91": (5, -20, 15, 91), "16x180": (16, -15, 15, 180),
                                                     "5x2048": (5, -20, 15, 2048)}[name]))


SCENES = {}


def scene(kind):
    if kind not in SCENES:
        if kind in ("room", "boxes"):
            v, t, obs = synth.tiny_room_scene(3, n_boxes=8 if kind == "room" else 90)
        elif kind == "ball":
            v, t, obs = synth.indoor_scene(5, n_spheres=1, n_boxes=0)
        else:
            v, t, obs = synth.indoor_scene(5, n_spheres={"5k": 9, "10k": 20, "64k": 120}[kind],
                                           n_boxes={"5k": 5, "10k": 9, "64k": 60}[kind])
        vc, tc = torch.from_numpy(v).cuda(), torch.from_numpy(t).cuda()
        P = synth.sample_free_pose(np.random.default_rng(1), obs, 64, upright=False)
        SCENES[kind] = (fgl.Scene(v, t), fgl.Lbvh(vc, tc), torch.from_numpy(P).cuda())
    return SCENES[kind]


@pytest.mark.parametrize("kind", ["room", "boxes", "ball", "5k", "10k", "64k"])
@pytest.mark.parametrize("name,rays", [("16x360", 5760), ("16x360", 140_000), ("16x360", 530_000), ("16x360", 4_300_000),
                                       ("16x180", 30_000), ("16x180", 300_000), ("5x2048", 60_000),
                                       ("5x91", 30_000),
                                       ("5x91", 60_000), ("5x91", 80_000), ("field4x4", 4000), ("field3x11", 70_000),
                                       ("field7x8", 70_000), ("field1x27", 5000), ("field1x28", 5000)])
def test_rule(kind, name, rays):
    sc, lb, poses = scene(kind)
    se = sensor(name)
    envs = -(-rays // se.n_rays)
    P = poses.repeat(-(-envs // 64), 1, 1)[:envs].contiguous()
    n = envs * se.n_rays

    def out():
        return torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")

    for near in (0.0, 0.5):
        ref, got, static = out(), out(), out()
        fgl.cast_batched([(sc, se, P, 60.0, *ref, near)], fgl.BatchOpts(tri_mode=1))
        fgl.cast_batched([(sc, se, P, 60.0, *got, near)])
        fgl.cast_batched_static([(sc, se, P, 60.0, *static, near)])
        runs = [got, static, lb.cast(se, P, 60.0, min_range=near)]
        if near == 0.0:
            runs += [fgl.cast(sc, se, P, 60.0), fgl.cast_opts(sc, se, P, 60.0, fgl.BatchOpts())]
        fgl.sync()
        for r, i in runs:
            assert torch.equal(r.reshape(-1), ref[0]) and torch.equal(i.reshape(-1), ref[1])
    assert lb.stats()["overflow"] == 0
