"""The density kernel's two evaluation forms and its splits, against the FP64
oracle within the oracle's per-voxel tolerance (the bound of the random-Gaussian
parity test): Gaussians on both sides of the steepness limit and far along a
row, grids of few and of many tiles (candidates split over eight or four, four
or one warps), partial tiles, tiles with fewer candidates than a batch and with
a batch more or less; and masks that follow from the returned density exactly
when theta is a voxel's own density."""

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


def run(g, origin, h, dims, theta, tile):
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in g]
    D, occ, surf, _ = fgl.gaussian_density(*t, origin, h, dims, theta=theta, tile=tile)
    torch.cuda.synchronize()
    return D.cpu().numpy(), occ.cpu().numpy(), surf.cpu().numpy()


def gaussians(rng, n, extent, smin, smax):
    return (rng.uniform(-0.1, extent + 0.1, (n, 3)).astype(np.float32),
            np.exp(rng.uniform(np.log(smin), np.log(smax), (n, 3))).astype(np.float32),
            rng.standard_normal((n, 4)).astype(np.float32), rng.uniform(0.2, 1.0, n).astype(np.float32))


# (tile, voxel, dims, Gaussians, smallest and largest scale): flat rows only,
# both forms, steep rows only; 2,744 tiles take the split of large grids
@pytest.mark.parametrize("tile,h,dims,n,smin,smax", [
    (8, 0.02, (24, 17, 9), 300, 0.05, 0.2),
    (8, 0.05, (33, 16, 23), 500, 0.01, 0.2),
    (8, 0.10, (16, 16, 16), 200, 0.01, 0.04),
    (8, 0.03, (112, 110, 106), 400, 0.01, 0.15),
    (4, 0.05, (13, 9, 7), 300, 0.01, 0.2),
    (4, 0.04, (56, 55, 54), 300, 0.01, 0.15),
    (8, 0.05, (8, 8, 8), 31, 0.02, 0.2), (8, 0.05, (8, 8, 8), 33, 0.02, 0.2), (8, 0.05, (8, 8, 8), 257, 0.02, 0.2),
    (4, 0.05, (4, 4, 4), 1, 0.02, 0.2), (4, 0.05, (4, 4, 4), 129, 0.02, 0.2)])
def test_forms_and_splits_vs_oracle(tile, h, dims, n, smin, smax):
    rng = np.random.default_rng(tile * 1000 + n + dims[0])
    g = gaussians(rng, n, h * np.array(dims), smin, smax)
    origin = (0.01, -0.02, 0.03)
    D, occ, surf = run(g, origin, h, dims, 0.5, tile)
    Do, Ao = oracle.density(*g, origin, h, dims, tile)
    tol = oracle.density_tolerance(Do, Ao)
    assert np.all(np.abs(D.astype(np.float64) - Do) <= tol)
    occ_g, surf_g = oracle.occupancy(D.astype(np.float64), 0.5)
    assert np.array_equal(occ, occ_g) and np.array_equal(surf, surf_g)
    # theta on a voxel's own density: that voxel (and others close to it) are
    # summed voxel by voxel, within the same tolerance, and the masks follow
    for v in rng.choice(D.size, 3, replace=False):
        theta = float(D.reshape(-1)[v])
        E, occ, surf = run(g, origin, h, dims, theta, tile)
        assert np.all(np.abs(E.astype(np.float64) - Do) <= tol)
        occ_g, surf_g = oracle.occupancy(E.astype(np.float64), np.float64(np.float32(theta)))
        assert np.array_equal(occ, occ_g) and np.array_equal(surf, surf_g)


def test_far_thin_gaussian_adds_no_nan():
    """Thin, long, tilted Gaussians whose rows lie hundreds of standard
    deviations from the ridge: every exponential underflows or the candidate
    is evaluated voxel by voxel; no infinity or NaN appears."""
    n = 64
    rng = np.random.default_rng(5)
    mu = rng.uniform(0, 1, (n, 3)).astype(np.float32)
    scale = np.tile(np.array([0.002, 0.003, 0.5], np.float32), (n, 1))
    q = rng.standard_normal((n, 4)).astype(np.float32)
    al = np.ones(n, np.float32)
    for h in (0.002, 0.02, 0.05):
        dims = (20, 20, 20)
        D, _, _ = run((mu, scale, q, al), (0.0, 0.0, 0.0), h, dims, 0.5, 8)
        assert np.all(np.isfinite(D)) and np.all(D >= 0)


# a tile shared by a cluster's blocks (more than two batches a warp, and one
# less), and more voxels at theta than are summed at once: Gaussians mirrored
# about the tile's middle planes give eight voxels the same density up to
# rounding
@pytest.mark.parametrize("tile,n", [(8, 512), (8, 520), (8, 4096), (4, 256), (4, 264), (4, 2048)])
def test_shared_tiles_and_equal_voxels(tile, n):
    rng = np.random.default_rng(n + tile)
    h = 0.05
    L = h * tile
    m, s, q, a = gaussians(rng, n // 8, L / 2, 0.02, 0.2)
    q[:] = (1, 0, 0, 0)
    sign = np.array([[x, y, z] for x in (1, -1) for y in (1, -1) for z in (1, -1)], np.float32)
    g = (((m - L / 2)[None] * sign[:, None] + L / 2).reshape(-1, 3).astype(np.float32), np.tile(s, (8, 1)),
         np.tile(q, (8, 1)), np.tile(a, 8))
    dims = (tile, tile, tile)
    Do, Ao = oracle.density(*g, (0.0, 0.0, 0.0), h, dims, tile)
    tol = oracle.density_tolerance(Do, Ao)
    D, _, _ = run(g, (0.0, 0.0, 0.0), h, dims, 0.5, tile)
    assert np.all(np.abs(D.astype(np.float64) - Do) <= tol)
    theta = float(D.reshape(-1)[tile * tile + 1])
    E, occ, surf = run(g, (0.0, 0.0, 0.0), h, dims, theta, tile)
    assert np.all(np.abs(E.astype(np.float64) - Do) <= tol)
    occ_g, surf_g = oracle.occupancy(E.astype(np.float64), np.float64(np.float32(theta)))
    assert np.array_equal(occ, occ_g) and np.array_equal(surf, surf_g)
