"""The density kernel's splits over grids from nearly empty to dense, on either side
of the mean candidates a tile at which one takes over from another (2,744 tiles and
more, partial ones among them, most of them nobody's in the first): against the FP64
oracle within its per-voxel tolerance, with exact zeros where no candidate is, in both
tile sizes."""

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


@pytest.mark.parametrize("n,smax,tile,least,most", [(3, 0.1, 8, 0, 1), (700, 0.12, 8, 1, 32), (900, 0.45, 8, 32, 1024),
                                                    (9000, 0.6, 8, 1024, 1 << 30), (40, 0.05, 4, 0, 1)])
def test_sparse_to_dense(n, smax, tile, least, most):
    rng = np.random.default_rng(n)
    h, dims = 0.03, (112, 110, 106) if tile == 8 else (56, 55, 54)
    g = [rng.uniform(0, 1, (n, 3)) * h * np.array(dims), np.exp(rng.uniform(np.log(0.3 * smax), np.log(smax), (n, 3))),
         rng.standard_normal((n, 4)), rng.uniform(0.2, 1, n) / (1.0 + n / 500.0)]
    g = [np.ascontiguousarray(a, np.float32) for a in g]
    Do, Ao = oracle.density(*g, (0.0, 0.0, 0.0), h, dims, tile)
    theta = float(np.float32(0.3 * Do.max()))
    D, occ, surf, st = fgl.gaussian_density(*[torch.from_numpy(a).cuda() for a in g], (0.0, 0.0, 0.0), h, dims, theta=theta, tile=tile)
    assert least <= st["n_pairs"] / st["n_tiles"] < most and st["n_tiles"] >= 2432
    D = D.cpu().numpy()
    assert np.all(np.abs(D.astype(np.float64) - Do) <= oracle.density_tolerance(Do, Ao))
    assert np.all(D[Do == 0] == 0)
    occ_g, surf_g = oracle.occupancy(D.astype(np.float64), np.float64(theta))
    assert np.array_equal(occ.cpu().numpy(), occ_g) and np.array_equal(surf.cpu().numpy(), surf_g)
