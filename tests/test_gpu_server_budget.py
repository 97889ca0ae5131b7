"""The server's budget counts every byte a resident scene holds on the device: its
node and triangle records and the top cut (32 boxes of 32 bytes and up to 24
triangles) behind them."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
fgl = pytest.importorskip("paper_2509_17390_gb300")


@pytest.mark.parametrize("n", [3, 20_000])
def test_resident_scene_is_counted_whole(n):
    rng = np.random.default_rng(n)
    v = (rng.uniform(0, 4, (n, 1, 3)) + 0.1 * rng.standard_normal((n, 3, 3))).reshape(-1, 3).astype(np.float32)
    sc = fgl.Scene(v, np.arange(3 * n, dtype=np.int32).reshape(n, 3))
    st = sc.stats()
    srv = fgl.Server(hbm_budget_bytes=1 << 30)
    before = srv.stats()["device_bytes"]
    sid = srv.add_scene(sc)
    held = srv.stats()["device_bytes"] - before
    assert st["node_bytes"] + st["tri_bytes"] + 32 * 32 <= held <= st["node_bytes"] + st["tri_bytes"] + 32 * 32 + 24 * 48 + 256
    tid = srv.add_sensor(fgl.Sensor.from_table(synth.grid_sensor(4, -10, 10, 90)))
    P = np.eye(3, 4, dtype=np.float32)[None].copy()
    P[:, :, 3] = 2.0
    r, i = np.empty(360, np.float32), np.empty(360, np.int32)
    srv.wait(srv.submit(sid, tid, P, 30.0, r, i))
    assert srv.stats()["device_bytes"] - before == held      # the request's own bytes are given back
    srv.close()
