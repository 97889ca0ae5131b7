"""The masks do not hang on how a tile's candidates are split or evaluated.

A grid and the same grid continued by empty tiles have the same candidates a tile
but go to kernels of different splits (few tiles and many, a mean of few and of many
candidates): with theta at a voxel's own density the occupancy and surface masks of
the common voxels are equal, and so is the density of that voxel, which is summed
again in candidate order.  Over usual Gaussians, thin ones at every angle (whose
exponents are sums of terms thousands of times as large), very many equal ones (whose
rounding errors all point one way) and both tile sizes.  And where theta is 0 or of the
size of what underflows, a voxel is occupied by the 64-bit density alone.

A voxel's sum in candidate order is what comes back for it when theta is its density;
just below that sum the voxel is occupied, at it not, whatever its first density was."""

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


def gaussians(kind, L, n):
    rng = np.random.default_rng(n)
    q = rng.standard_normal((n, 4))
    mu = rng.uniform(0, L, (n, 3))
    al = rng.uniform(0.3, 1.0, n)
    if kind == "usual":
        s = np.exp(rng.uniform(np.log(0.01), np.log(0.15), (n, 3)))
    elif kind == "equal":
        mu, s, q = np.tile(0.4 * L, (n, 1)), np.tile([0.1, 0.12, 0.09], (n, 1)), np.tile([1.0, 0, 0, 0], (n, 1))
        al = np.full(n, 0.7 / n ** 0.5)
    else:
        s = np.tile({"disc": [0.003, 0.5, 0.5], "thinner": [0.0005, 0.5, 0.5], "needle": [0.003, 0.003, 0.6]}[kind], (n, 1))
    return [torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda() for a in (mu, s, q, al)]


@pytest.mark.parametrize("kind,n,tile", [("usual", 2000, 8), ("usual", 130_000, 8), ("usual", 2000, 4), ("disc", 300, 8),
                                         ("disc", 300, 4), ("thinner", 300, 8), ("needle", 400, 8), ("needle", 400, 4),
                                         ("equal", 16_000, 8), ("equal", 40_000, 8), ("equal", 120_000, 8), ("equal", 30_000, 4)])
def test_masks_of_a_grid_and_its_continuation(kind, n, tile):
    h, d = 0.05, 3 * tile
    g = gaussians(kind, np.array([d, d, d]) * h, n)
    small, large = (d, d, d), (d, d, 300 * tile)          # 27 tiles and 2,700
    run = lambda dims, theta: fgl.gaussian_density(*g, (0.0, 0.0, 0.0), h, dims, theta=theta, tile=tile)
    D = run(small, 1e30)[0].cpu().numpy()
    rng = np.random.default_rng(3)
    for v in rng.choice(np.flatnonzero(D > 1e-4 * D.max()), 16):
        theta = float(D.reshape(-1)[v])
        a, b = run(small, theta), run(large, theta)
        inner = slice(0, d - 1)                            # the surface mask looks one voxel further
        assert torch.equal(a[1], b[1][:d])
        assert torch.equal(a[2][inner], b[2][inner])
        assert float(a[0].reshape(-1)[v]) == float(b[0][:d].reshape(-1)[v])
        for D1, occ in (a[:2], b[:2]):
            assert torch.equal(occ.bool(), D1 > theta)


@pytest.mark.parametrize("kind,n,tile", [("usual", 2000, 8), ("disc", 300, 8), ("disc", 300, 4), ("thinner", 300, 8),
                                         ("needle", 400, 8), ("needle", 400, 4), ("equal", 16_000, 8), ("equal", 40_000, 4)])
def test_masks_follow_the_sum_in_candidate_order(kind, n, tile):
    h, dims = 0.05, (3 * tile,) * 3
    g = gaussians(kind, np.array(dims) * h, n)
    run = lambda theta: [a.reshape(-1) for a in fgl.gaussian_density(*g, (0.0, 0.0, 0.0), h, dims, theta=theta, tile=tile)[:2]]
    D = run(1e30)[0].cpu().numpy()
    rng = np.random.default_rng(5)
    for v in rng.choice(np.flatnonzero(D > 1e-3 * D.max()), 40):
        v = int(v)
        s = float(run(float(D[v]))[0][v])
        at, below = run(s), run(float(np.nextafter(np.float32(s), np.float32(0))))
        assert float(at[0][v]) == s and int(at[1][v]) == 0
        assert float(below[0][v]) == s and int(below[1][v]) == 1


@pytest.mark.parametrize("tile", [8, 4])
def test_theta_below_what_underflows(tile):
    rng = np.random.default_rng(3)
    n, h, dims = 40, 0.05, (80, 80, 80)
    g = [rng.uniform(0, 4, (n, 3)), np.exp(rng.uniform(np.log(0.01), np.log(0.3), (n, 3))), rng.standard_normal((n, 4)),
         rng.uniform(0.2, 1, n)]
    g = [np.ascontiguousarray(a, np.float32) for a in g]
    Do, _ = oracle.density(*g, (0.0, 0.0, 0.0), h, dims, tile)
    cu = [torch.from_numpy(a).cuda() for a in g]
    for theta in (0.0, 1e-45, 1e-40, 1e-37, 1e-30, 1e-20, 1e-14, 1e-11, 1e-9, 2e-9):
        t = float(np.float32(theta))
        D, occ, _, _ = fgl.gaussian_density(*cu, (0.0, 0.0, 0.0), h, dims, theta=theta, tile=tile)
        D, occ = D.cpu().numpy(), occ.cpu().numpy()
        assert np.array_equal(occ, (D > np.float32(theta)).astype(np.uint8))
        # an exponent is a sum of terms up to 6,000 here, ten roundings: 0.5% of the density at most;
        # a single-precision exponential underflows below 2^-126, a sum of 40 below 2^-120
        sure = (Do > 1.02 * t) & (Do > 2.0 ** -120)
        assert np.all(occ[sure] == 1)
        assert np.all(occ[(Do < 0.98 * t) & (t > 2.0 ** -120)] == 0)
        assert np.all(occ[Do < 2.0 ** -150] == 0) and int(occ.sum()) > 1000
