"""The record counts an LBVH's casts are checked against by the checked library:
the 8-wide form's node count is the number of nodes reached from its root, not
the capacity of their array."""

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


def mesh(seed, n):
    rng = np.random.default_rng(seed)
    v = (rng.uniform(0, 4, (n, 1, 3)) + 0.3 * rng.standard_normal((n, 3, 3))).reshape(-1, 3)
    return torch.from_numpy(v.astype(np.float32)).cuda(), torch.arange(3 * n, dtype=torch.int32).reshape(n, 3).cuda()


class Item(ctypes.Structure):   # a cast's item record: the node array and the record counts
    _fields_ = [("nodes", ctypes.c_void_p), ("between", ctypes.c_uint64 * 9), ("n_nodes", ctypes.c_uint32),
                ("n_tris", ctypes.c_uint32), ("rest", ctypes.c_uint64 * 3)]


@pytest.mark.parametrize("n", [1, 2, 7, 9, 257, 5000])
def test_wide_node_count_is_exact(n):
    v, t = mesh(3, n)
    lb = fgl.Lbvh(v, t)
    lb.rebuild(v, t)
    item = fgl.lib()["_ZN3fgl9lbvh_itemEPK10fgl_lbvh_s"]
    item.restype, item.argtypes = Item, [ctypes.c_void_p]
    it = item(lb.handle)

    class View:
        __cuda_array_interface__ = {"shape": (it.n_nodes, 64), "typestr": "<i4", "data": (it.nodes, False), "version": 2}
    w = torch.as_tensor(View(), device="cuda").cpu().numpy().view(np.uint32)
    reached, tris = {0}, 0
    todo = [0]
    while todo:
        k = todo.pop()
        assert k < it.n_nodes
        kids = bin(int(w[k, 3]) & 0xFF).count("1")
        tris += sum(bin(int(x) & 0xFFFFFF).count("1") for x in w[k, 56:])
        for c in range(int(w[k, 4]), int(w[k, 4]) + kids):
            assert c not in reached
            reached.add(c)
            todo.append(c)
    assert len(reached) == it.n_nodes and tris == it.n_tris == n
