"""The tiled shells and the warp-wide mesh emission at the sizes where they can
go wrong: rows of one word, of whole tiles of words and of one more, tiles cut
off on every side, bands up to the tiled limit of six shells and one past it
(phi, signs and shells bit for bit the oracle's); sample grids with a word's
last bit at a cube, a chunk of 256 words and one more, more words than are
counted one a thread, and strides (triangles exact, vertices within the
oracle's tolerance, normals as one by one)."""

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("L", [1, 5, 6, 7])
@pytest.mark.parametrize("shape", [(8, 8, 32), (9, 7, 33), (17, 16, 256), (3, 25, 257), (16, 9, 289)])
def test_shells_at_tile_edges(shape, L):
    rng = np.random.default_rng(sum(shape) + L)
    V = (rng.random(shape) < 0.02).astype(np.uint8)
    V[shape[0] // 2, :, : shape[2] // 2] = 1
    h = 0.02
    phi, out, sh, st = fgl.tsdf(cu(V), h, L * h, outside=True, shell=True)
    phi_o, out_o, p_o = oracle.tsdf(V, h, L * h)
    assert st["n_layers"] == oracle.band_layers(h, L * h)
    assert np.array_equal(out.cpu().numpy(), out_o) and np.array_equal(sh.cpu().numpy(), p_o)
    assert np.array_equal(phi.cpu().numpy().view(np.uint32), phi_o.view(np.uint32))
    alone = fgl.tsdf(cu(V), h, L * h)[0]                      # without the other outputs
    assert torch.equal(alone, phi)


@pytest.mark.parametrize("shape,step", [((2, 2, 2), 1), ((3, 5, 33), 1), ((4, 4, 64), 1), ((16, 16, 30), 1),
                                        ((1, 256, 32), 1), ((2, 129, 31), 1), ((7, 11, 130), 2), ((258, 257, 33), 1)])
def test_emission_at_word_and_chunk_edges(shape, step):
    rng = np.random.default_rng(sum(shape))
    phi = rng.standard_normal(shape).astype(np.float32)
    if phi.size > 1 << 20:
        phi = np.abs(phi) + np.float32(0.1)                   # crossings at a few places, the last word among them
        phi[rng.integers(0, shape[0], 300), rng.integers(0, shape[1], 300), rng.integers(0, shape[2], 300)] *= -1
        phi[-1, -1, -1] = -0.3
    o, h = (0.1, -0.2, 0.3), 0.05
    v, t, n = fgl.marching_tets(cu(phi), o, h, step=step, normals=True)
    torch.cuda.synchronize()
    v_o, t_o, n_o = oracle.marching_tets(phi, o, h, step=step, normals=True)
    assert np.array_equal(t.cpu().numpy(), t_o) and v.shape[0] == len(v_o)
    assert np.max(np.abs(v.cpu().numpy() - v_o), initial=0.0) <= oracle.vertex_tolerance(v_o, h * step)
    bare = fgl.marching_tets(cu(phi), o, h, step=step)
    assert torch.equal(bare[0], v) and torch.equal(bare[1], t)
    if len(v_o):
        clear = np.linalg.norm(n_o, axis=1) > 0.5             # the gradient is not zero there
        assert np.max(np.abs(n.cpu().numpy()[clear] - n_o[clear]), initial=0.0) < 1e-3
