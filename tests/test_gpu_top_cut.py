"""Packets start from a cut through the top of the tree: scenes whose cut is
the root's children alone (one to forty triangles), has leaf triangles of its
own (large triangles among small ones) or more of them than a cut holds (no
cut), and whose boxes nearly all meet every packet (nested shells: on from the
root).  Returns equal the one-thread-a-ray form's, bit for bit, for both
widths, batched and alone, with and without a minimum range, and after the
scene was evicted and uploaded again."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


def triangles(rng, kind):
    if kind.startswith("few"):
        c = rng.uniform(-3, 3, (int(kind[3:]), 1, 3))
        return c + rng.uniform(-1, 1, (len(c), 3, 3))
    small = rng.uniform(-4, 4, (4000, 1, 3)) + rng.uniform(-0.05, 0.05, (4000, 3, 3))
    if kind.startswith("large"):
        return np.concatenate([small, rng.uniform(-12, 12, (int(kind[5:]), 3, 3))])
    # nested shells around the sensor: the boxes of every part of a shell that
    # spans it overlap
    d = rng.standard_normal((6000, 3, 3))
    d /= np.linalg.norm(d, axis=2, keepdims=True)
    return d * rng.uniform(2, 6, (6000, 1, 1))


@pytest.mark.parametrize("width", [4, 8])
@pytest.mark.parametrize("kind", ["few1", "few3", "few9", "few40", "large3", "large20", "large400", "shells"])
def test_cuts(kind, width):
    rng = np.random.default_rng(len(kind) * 10 + width)
    v = triangles(rng, kind).astype(np.float32).reshape(-1, 3)
    sc = fgl.Scene(v, np.arange(len(v), dtype=np.int32).reshape(-1, 3), width=width)
    se = fgl.Sensor.from_table(synth.grid_sensor(16, -30, 30, 180))
    P = np.zeros((5, 3, 4), np.float32)
    P[:, :, :3] = synth.random_rotation(rng, 5)
    P[:, :, 3] = rng.uniform(-2, 2, (5, 3))
    P[0, :, 3] = 0.0
    pose = torch.from_numpy(P).cuda()
    n = 5 * se.n_rays

    def out():
        return torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")

    for near in (0.0, 1.5):
        want, got = out(), out()
        fgl.cast_batched([(sc, se, pose, 30.0, *want, near)], fgl.BatchOpts(tri_mode=1))
        fgl.cast_batched([(sc, se, pose, 30.0, *got, near)])
        fgl.sync()
        assert torch.equal(want[0], got[0]) and torch.equal(want[1], got[1])
        if near == 0.0:
            alone = fgl.cast(sc, se, pose, 30.0)
            fgl.sync()
            assert torch.equal(want[0], alone[0].reshape(-1)) and torch.equal(want[1], alone[1].reshape(-1))
    sc.evict()
    sc.upload()
    got = out()
    fgl.cast_batched([(sc, se, pose, 30.0, *got, 1.5)])
    fgl.sync()
    assert torch.equal(want[0], got[0]) and torch.equal(want[1], got[1])
