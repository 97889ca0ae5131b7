"""fgl_apply_sensor_effects over the shapes where its blocks and vector
accesses can go wrong: arrays shorter than four returns, one more or less than
a block's 1,024, pointers that are not 16-byte aligned, environments of one ray
and blocks that span many environments -- against the FP64 oracle within the
parity test's bounds, and bitwise equal to the aligned call."""

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")

FX = dict(seed=0x1234567890, step=7, env_offset=11, drop_prob=0.2, sigma0=0.02, sigma1=0.003)


def apply(t, i, n_env, shift):
    n = len(t)
    r = torch.zeros(n + 4, dtype=torch.float32, device="cuda")[shift:shift + n]
    k = torch.zeros(n + 4, dtype=torch.int32, device="cuda")[shift:shift + n]
    r.copy_(torch.from_numpy(t))
    k.copy_(torch.from_numpy(i))
    fgl.apply_sensor_effects(r, k, n_env, max_range=30.0, **FX)
    torch.cuda.synchronize()
    return r.cpu().numpy(), k.cpu().numpy()


@pytest.mark.parametrize("n_env,n_rays", [(1, 1), (3, 1), (1, 5), (1, 1023), (1, 1024), (1, 1025), (1025, 1), (341, 3), (2, 1024),
                                          (7, 333), (5, 2049)])
def test_shapes_and_alignment(n_env, n_rays):
    rng = np.random.default_rng(n_env * 7 + n_rays)
    n = n_env * n_rays
    t = rng.uniform(0.1, 30.0, n).astype(np.float32)
    i = np.where(rng.random(n) < 0.8, rng.integers(0, 1000, n), -1).astype(np.int32)
    t[i < 0] = 30.0
    ref = apply(t, i, n_env, 0)
    for shift in (1, 2, 3):
        got = apply(t, i, n_env, shift)
        assert np.array_equal(ref[0], got[0]) and np.array_equal(ref[1], got[1])
    tn, inn, _ = oracle.sensor_effects(t, i, n_env, max_range=30.0, **FX)
    assert np.array_equal(ref[1], inn)
    tol = 6e-7 * np.maximum(np.abs(t), 1) + 5e-6 * (FX["sigma0"] + FX["sigma1"] * t)
    assert np.all(np.abs(ref[0].astype(np.float64) - tn) <= tol)
