"""The stable radix sort behind the LBVH and the pair lists: the LBVH's export
lists its triangles by Morton code, equal codes in input order, for arrays
around a slice (2,048 keys; 4,096 from 1,245,184 keys on) and its remainders,
and for keys that are all equal."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


def morton(c):
    f = np.float32
    lo, hi = c.min(0), c.max(0)
    q = np.zeros(c.shape, f)
    for a in range(3):
        if hi[a] > lo[a]:
            q[:, a] = (c[:, a] - lo[a]) / (hi[a] - lo[a]) * f(1024)
    u = np.clip(q, f(0), f(1023)).astype(np.uint32)
    m = np.zeros(len(c), np.uint32)
    for b in range(10):
        for a in range(3):
            m |= ((u[:, a] >> np.uint32(b)) & np.uint32(1)) << np.uint32(3 * b + 2 - a)
    return m


@pytest.mark.parametrize("n", [2, 255, 2047, 2048, 2049, 70_001, 1_245_183, 1_245_184, 1_300_003])
@pytest.mark.parametrize("cells", [3, 1000])
def test_triangles_in_morton_order(n, cells):
    rng = np.random.default_rng(n + cells)
    # centroids on a lattice of exact floats (many equal codes when it is coarse)
    c = (rng.integers(0, cells, (n, 3)) / 8.0).astype(np.float32)
    c[0], c[-1] = 0.0, cells / 8.0
    d = np.float32(2.0 ** -6)
    v = np.stack([c - [d, 0, 0], c + [d, 0, 0], c + [0, d, 0]], 1)
    v[:, 2, 1] = c[:, 1]                            # flat in y: the box's middle is c
    lo, hi = v.min(1), v.max(1)
    mid = (np.float32(0.5) * lo + np.float32(0.5) * hi).astype(np.float32)
    tris = np.arange(3 * n, dtype=np.int32).reshape(n, 3)
    lb = fgl.Lbvh(torch.from_numpy(v.reshape(-1, 3).astype(np.float32)).cuda(), torch.from_numpy(tris).cuda())
    _, rec = lb.export()
    ids = rec[:, 3].copy().view(np.int32)
    assert np.array_equal(ids, np.argsort(morton(mid), kind="stable"))
