"""A scene's device buffer -- nodes, triangles, the top cut's triangles and the
cut in one allocation -- on both sides of the size up to which it is staged for one
copy, and for scenes without a cut: evicted and uploaded again, both widths, casts
return what the lane-serial form returns (which reads no cut)."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


@pytest.mark.parametrize("width", [8, 4])
@pytest.mark.parametrize("n", [1, 5, 400, 1100, 1500, 3000, 40_000])   # staged up to some 1,200 to 1,900 triangles
def test_buffer_parts(n, width):
    rng = np.random.default_rng(n + width)
    v = (rng.uniform(-4, 4, (n, 1, 3)) + 0.2 * rng.standard_normal((n, 3, 3))).reshape(-1, 3).astype(np.float32)
    sc = fgl.Scene(v, np.arange(3 * n, dtype=np.int32).reshape(n, 3), width=width)
    se = fgl.Sensor.from_table(synth.grid_sensor(16, -30, 30, 360))
    P = np.zeros((92, 3, 4), np.float32)                   # 529,920 rays: packets in any scene
    P[:, :, :3] = synth.random_rotation(rng, 92)
    P[:, :, 3] = rng.uniform(-3, 3, (92, 3))
    pose = torch.from_numpy(P).cuda()
    m = 92 * se.n_rays
    want = torch.empty(m, device="cuda"), torch.empty(m, dtype=torch.int32, device="cuda")
    fgl.cast_batched([(sc, se, pose, 30.0, *want)], fgl.BatchOpts(tri_mode=1))
    for _ in range(2):
        got = fgl.cast(sc, se, pose, 30.0)
        batch = torch.empty_like(want[0]), torch.empty_like(want[1])
        fgl.cast_batched([(sc, se, pose, 30.0, *batch)])
        fgl.sync()
        for r, i in (got, batch):
            assert torch.equal(r, want[0]) and torch.equal(i, want[1])
        sc.evict()
        sc.upload()
