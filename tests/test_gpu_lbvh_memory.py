"""An LBVH of a mesh that fits the device's free memory only without the 8-wide form
(139 of some 360 bytes a triangle) is built without it, and returns what the whole
one returns; with room again, the next build makes it."""

import ctypes

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


class Item(ctypes.Structure):   # a cast's item record: the node array comes first
    _fields_ = [("nodes", ctypes.c_void_p), ("rest", ctypes.c_uint64 * 13)]


def wide_nodes(lb):
    item = fgl.lib()["_ZN3fgl9lbvh_itemEPK10fgl_lbvh_s"]
    item.restype, item.argtypes = Item, [ctypes.c_void_p]
    return item(lb.handle).nodes


def test_built_without_the_wide_form():
    n = 3_000_000
    g = torch.Generator(device="cuda").manual_seed(1)
    v = (torch.rand((n, 1, 3), generator=g, device="cuda") * 4 +
         0.02 * torch.randn((n, 3, 3), generator=g, device="cuda")).reshape(-1, 3)
    t = torch.arange(3 * n, dtype=torch.int32, device="cuda").reshape(n, 3)
    P = np.zeros((20, 3, 4), np.float32)
    P[:, :, :3] = synth.random_rotation(np.random.default_rng(1), 20)
    P[:, :, 3] = 2.0
    pose = torch.from_numpy(P).cuda()
    sensors = [fgl.Sensor.from_table(x) for x in (synth.grid_sensor(16, -15, 15, 360), synth.rosette_sensor(2000, 1))]
    lb = fgl.Lbvh(v, t)
    assert wide_nodes(lb)
    want = [lb.cast(se, pose, 20.0) for se in sensors]
    got = [(torch.empty_like(r), torch.empty_like(i)) for r, i in want]
    fgl.sync()
    lb.close()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - n * 290, dtype=torch.uint8, device="cuda")   # 218 B without, 357 with the wide form
    try:
        lb = fgl.Lbvh(v, t)
        assert not wide_nodes(lb)
        for se, (r, i) in zip(sensors, got):
            lb.cast(se, pose, 20.0, out_range=r, out_tri=i)
        fgl.sync()
    finally:
        del hog
        torch.cuda.empty_cache()
    for a, b in zip(want, got):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    lb.rebuild(v, t)
    assert wide_nodes(lb)
    r, i = lb.cast(sensors[0], pose, 20.0)
    fgl.sync()
    assert torch.equal(r, want[0][0]) and torch.equal(i, want[0][1])
    assert lb.stats()["overflow"] == 0
