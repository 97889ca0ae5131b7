"""An LBVH after a rebuild that was refused: its arrays hold no tree, so it is
neither cast nor exported until a good rebuild revives it."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


def mesh(seed, n):
    rng = np.random.default_rng(seed)
    v = (rng.uniform(0, 4, (n, 1, 3)) + 0.3 * rng.standard_normal((n, 3, 3))).reshape(-1, 3)
    return torch.from_numpy(v.astype(np.float32)).cuda(), torch.arange(3 * n, dtype=torch.int32).reshape(n, 3).cuda()


@pytest.mark.parametrize("n", [1, 300, 301])    # 300: the arrays stay, others: made anew
def test_refused_rebuild_leaves_nothing_to_cast(n):
    v, t = mesh(1, 300)
    lb = fgl.Lbvh(v, t)
    se = fgl.Sensor.from_table(synth.grid_sensor(16, -15, 15, 90))
    P = torch.eye(3, 4, device="cuda")[None].repeat(4, 1, 1)
    P[:, :, 3] = 2.0
    want = lb.cast(se, P, 20.0)
    fgl.sync()
    bv, bt = mesh(2, n)
    bt[0, 1] = bv.shape[0]                      # a vertex id out of range
    for _ in range(2):
        with pytest.raises(fgl.FglError) as e:
            lb.rebuild(bv, bt)
        assert e.value.status == fgl.FGL_ERR_INVALID
        with pytest.raises(fgl.FglError) as e:
            lb.cast(se, P, 20.0)
        assert e.value.status == fgl.FGL_ERR_INVALID
        with pytest.raises(fgl.FglError):
            lb.export()
    lb.rebuild(v, t)
    got = lb.cast(se, P, 20.0)
    fgl.sync()
    assert torch.equal(want[0], got[0]) and torch.equal(want[1], got[1])
    assert lb.export()[1].shape == (300, 12)
