"""The LBVH's two casts -- packets over the 8-wide nodes, other rays one by one
over the binary tree -- return what the host-built tree returns, bit for bit:
sensors of both kinds on meshes of one triangle to several blocks of them, with
and without a minimum range -- and each goes to its own kernel."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


def kernels_of(call):
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        call()
        torch.cuda.synchronize()
    return [e.key for e in p.key_averages()]


@pytest.mark.parametrize("n", [1, 2, 300, 4000])
def test_rays_one_by_one_take_the_binary_tree(n):
    rng = np.random.default_rng(n)
    v = (rng.uniform(0, 4, (n, 1, 3)) + 0.3 * rng.standard_normal((n, 3, 3))).reshape(-1, 3).astype(np.float32)
    t = np.arange(3 * n, dtype=np.int32).reshape(n, 3)
    sc, lb = fgl.Scene(v, t), fgl.Lbvh(torch.from_numpy(v).cuda(), torch.from_numpy(t).cuda())
    P = np.zeros((40, 3, 4), np.float32)
    P[:, :, :3] = synth.random_rotation(rng, 40)
    P[:, :, 3] = rng.uniform(0, 4, (40, 3))
    pose = torch.from_numpy(P).cuda()
    for tab, binary in ((synth.rosette_sensor(3000, 1), True), (synth.grid_sensor(1, 0, 0, 5), True),
                        (synth.grid_sensor(16, -15, 15, 360), False)):
        se = fgl.Sensor.from_table(tab)
        for near in (0.0, 0.4):
            got = lb.cast(se, pose, 30.0, min_range=near)
            want = torch.empty_like(got[0]), torch.empty_like(got[1])
            fgl.cast_batched([(sc, se, pose, 30.0, *want, near)], fgl.BatchOpts(tri_mode=1))
            fgl.sync()
            assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        names = " ".join(kernels_of(lambda: lb.cast(se, pose, 30.0)))
        if names:                                   # where the profiler sees kernels
            assert ("k_lbvh_cast" in names) == binary, names
    assert lb.stats()["overflow"] == 0
