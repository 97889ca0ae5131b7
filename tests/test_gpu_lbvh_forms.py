"""The LBVH's block-local build and its wide form over the sizes where they can
go wrong: meshes of one to nine triangles (leaf runs only), one more or less
than a block of 256 leaves and of several, all triangles at one place (equal
codes: the hierarchy follows positions) and along a line (long chains).  The
exported tree's boxes nest and hold each triangle once, its depth is exact,
and casts with and without a minimum range return what the host-built wide BVH
returns, bit for bit."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


def soup(rng, n, layout):
    if layout == "room":
        c = rng.uniform(0, 4, (n, 3))
    elif layout == "point":
        c = np.full((n, 3), 2.0)
    else:
        c = np.stack([2.0 ** -np.arange(n).clip(max=40), np.full(n, 2.0), np.full(n, 2.0)], 1)
    e = rng.standard_normal((n, 3, 3)) * 0.3
    if layout == "point":
        e -= 0.5 * (e.min(1, keepdims=True) + e.max(1, keepdims=True))   # boxes share their middle
    return (c[:, None, :] + e).astype(np.float32)


def depth_of(left, right):
    depth = np.zeros(len(left), np.int64)
    order = [0]
    for k in order:
        for c in (left[k], right[k]):
            if c >= 0:
                depth[c] = depth[k] + 1
                order.append(c)
    assert len(order) == len(left)
    return int(depth.max()) + 2


@pytest.mark.parametrize("layout", ["room", "point", "line"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 9, 255, 256, 257, 511, 513, 3000])
def test_sizes_and_layouts(n, layout):
    rng = np.random.default_rng(n)
    v = soup(rng, n, layout).reshape(-1, 3)
    t = np.arange(3 * n, dtype=np.int32).reshape(n, 3)
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    lb = fgl.Lbvh(cu(v), cu(t))
    lb.rebuild(cu(v), cu(t))
    nodes, rec = lb.export()
    assert np.array_equal(np.sort(rec[:, 3].copy().view(np.int32)), np.arange(n))
    st = lb.stats()
    if n > 1:
        w = nodes.view(np.uint32).reshape(-1, 16)
        f = w[:, :12].copy().view(np.float32)
        d = w[:, 12:].copy().view(np.int32)
        box = {0: f[:, 0:6], 1: f[:, 6:12]}
        tv = rec.reshape(-1, 3, 4)[:, :, :3]
        lo, hi = tv.min(1), tv.max(1)
        own = np.concatenate([np.minimum(f[:, 0:3], f[:, 6:9]), np.maximum(f[:, 3:6], f[:, 9:12])], 1)
        for side in (0, 1):
            ref = d[:, side]
            leaf = ref < 0
            assert np.all(box[side][leaf, :3] <= lo[~ref[leaf]]) and np.all(box[side][leaf, 3:] >= hi[~ref[leaf]])
            assert np.array_equal(box[side][~leaf], own[ref[~leaf]])
            assert np.array_equal(d[ref[~leaf], 2], np.nonzero(~leaf)[0])
        assert d[0, 2] == -1 and st["depth"] == depth_of(d[:, 0], d[:, 1])
    P = np.zeros((3, 3, 4), np.float32)
    P[:, :, :3] = synth.random_rotation(rng, 3)
    P[:, :, 3] = [[2, 2, 2], [0.5, 3, 1], [-5, 2, 2]]
    # packets of neighbouring rays, a spread sensor and one of a few rays (one thread a ray)
    for tab in (synth.grid_sensor(16, -40, 40, 90), synth.rosette_sensor(100, 1), synth.grid_sensor(1, 0, 0, 5)):
        se = fgl.Sensor.from_table(tab)
        sc = fgl.Scene(v, t)
        for near in (0.0, 0.6):
            r1, i1 = lb.cast(se, cu(P), 20.0, min_range=near)
            r2, i2 = torch.empty_like(r1), torch.empty_like(i1)
            fgl.cast_batched([(sc, se, cu(P), 20.0, r2, i2, near)], fgl.BatchOpts(tri_mode=1))
            fgl.sync()
            assert torch.equal(r1, r2) and torch.equal(i1, i2)
    assert lb.stats()["overflow"] == 0
