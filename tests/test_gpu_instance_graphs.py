"""A captured batch is not replayed for an instance scene with other bounds: an
object destroyed and built again with moved vertices has the array sizes, and
often the addresses, of the one before, while its bounding sphere is an argument
of the captured launch."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


@pytest.mark.parametrize("widths", [(8,), (8, 4)])   # one launch for all instances, a launch each
def test_graph_follows_an_object_rebuilt_in_place(widths):
    v, t, obs = synth.tiny_room_scene(4)
    scene, se = fgl.Scene(v, t), fgl.Sensor.from_table(synth.grid_sensor(16, -15, 15, 360))
    P = torch.from_numpy(synth.sample_free_pose(np.random.default_rng(6), obs, 6)).cuda()
    n = 6 * se.n_rays
    uv, ut = synth.icosphere_unit(2)
    IP = torch.eye(3, 4, device="cuda").repeat(6, len(widths), 1, 1)
    IP[:, :, :, 3] = P[:, None, :, 3]
    IP = IP.contiguous()
    stream = torch.cuda.Stream()
    r, i = torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")
    k = torch.empty(n, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()

    def cast(inst, graph):
        with torch.cuda.stream(stream):
            fgl.cast_batched([(scene, se, P, 60.0, r, i, 0.0, {"instances": inst, "instance_poses": IP, "out_instance": k})],
                             fgl.BatchOpts(use_graph=1) if graph else None)
            fgl.sync()
        return r.clone(), i.clone(), k.clone()

    seen = set()
    for shift in (0.0, 1.2, -0.9, 2.0, 0.0):
        # a small ball beside the sensor, then on its other side, and so on
        inst = [fgl.Scene((0.3 * uv + [0.7 + shift, 0.1 * j, 0.0]).astype(np.float32), ut, width=w)
                for j, w in enumerate(widths)]
        got, want = cast(inst, True), cast(inst, False)
        for a, b in zip(got, want):
            assert torch.equal(a, b), shift
        assert int((want[2] >= 0).sum()) > 0
        seen.add(int((want[2] >= 0).sum()))
        for s in inst:
            s.close()
    assert len(seen) > 1
