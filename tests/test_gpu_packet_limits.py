"""Launch shapes at the edge of a block's shared memory: options the batched
cast accepts are cast whichever kernel the sensor takes.  The kernel that walks
whole packets needs 12 bytes a thread and its queue's words beyond the per-ray
one, so a shape may fit the one and not the other."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


# dynamic bytes of the packet kernel at width 8: 48,896 and 49,024 (with its own
# words past 48 KiB), 232,448 (alone as much as a block may have)
@pytest.mark.parametrize("block,depth", [(64, 31), (32, 63), (256, 37)])
@pytest.mark.parametrize("width", [8, 4])
def test_shapes_at_the_limit(block, depth, width):
    v, t, _ = synth.indoor_scene(5, n_spheres=120, n_boxes=60)
    sc = fgl.Scene(v, t, width=width)
    se = fgl.Sensor.from_table(synth.grid_sensor(16, -15, 15, 360))
    rng = np.random.default_rng(block)
    P = np.zeros((40, 3, 4), np.float32)
    P[:, :, :3] = synth.random_rotation(rng, 40)
    P[:, :, 3] = rng.uniform(0.1, 0.9, (40, 3)) * [20, 15, 4]
    pose = torch.from_numpy(P).cuda()
    n = 40 * se.n_rays

    def cast(opts, call=None):
        r, i = torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")
        (call or fgl.cast_batched)([(sc, se, pose, 60.0, r, i)], opts)
        fgl.sync()
        return r, i

    ref = cast(fgl.BatchOpts(tri_mode=1))
    opts = fgl.BatchOpts(block_threads=block, stack_smem=depth)
    got = [cast(opts), cast(opts, fgl.cast_batched_static), fgl.cast_opts(sc, se, pose, 60.0, opts)]
    hr, hi = np.empty(n, np.float32), np.empty(n, np.int32)
    fgl.cast_batched_host([(sc, se, P, 60.0, hr, hi)], opts)
    got.append((torch.from_numpy(hr).cuda(), torch.from_numpy(hi).cuda()))
    fgl.sync()
    for r, i in got:
        assert torch.equal(r.reshape(-1), ref[0]) and torch.equal(i.reshape(-1), ref[1])
