"""Depth-first walk that asks for possible receivers before it looks for the
end of a chain's last segment: records, segments and candidates equal the
breadth-first form's (which always looks), on both sides of the rule -- few
receivers, many receivers with few rays, many with many rays -- at every depth,
for receivers at segment ends (just above roofs and ground, at walls), forward,
backward and with launches smaller than one warp."""
import dataclasses

import numpy as np
import pytest

from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def engine():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine as E
    return E


def _both(g, **kw):
    a = g.trace(keep_rejected=True, **kw).records()
    sa = dict(g.last_stats)
    b = g.trace(keep_rejected=True, breadth_first=True, **kw).records()
    sb = dict(g.last_stats)
    assert np.array_equal(a, b)
    assert sa["segments"] == sb["segments"]
    assert sa["candidates"] == sb["candidates"]
    return len(a)


@pytest.mark.parametrize("n_rx,n_rays", [(1, 1), (3, 33), (16, 100_000), (200, 2_000),
                                         (2000, 40_000), (2000, 4_300_000)])
def test_walk_equals_breadth_first(engine, n_rx, n_rays):
    rng = np.random.default_rng(n_rx)
    sc = S.district_scene(seed=3, n_veh=37, n_rx=max(n_rx, 2), depth=4)
    fr = sc.frame(5)
    rx = fr.rx_pos[:n_rx].copy()
    rx[::3, 2] = np.float32(0.01)   # where rays end: on the ground
    hi = np.arange(n_rx)[::5]
    if n_rx > 10:                   # and just above roofs
        v = sc.face_xyz.reshape(-1, 3)
        top = v[v[:, 2] > 5]
        rx[hi] = top[rng.integers(0, len(top), len(hi))] + np.float32([0, 0, 0.02])
    fr = dataclasses.replace(fr, rx_pos=rx, rx_vel=np.zeros_like(rx))
    g = engine.Scene(sc, max_rx=n_rx)
    g.update(fr)
    found = 0
    for depth in (range(5) if n_rays < 1_000_000 else (2, 4)):
        found += _both(g, n_rays=n_rays, max_depth=depth)
    assert found > 0 or n_rays < 100


def test_backward_walk_equals_breadth_first(engine):
    sc = S.district_scene(seed=3, n_veh=37, n_rx=500, depth=4)
    g = engine.Scene(sc)
    g.update(sc.frame(5))
    ids = torch.arange(0, 500, 71, dtype=torch.int32, device="cuda")
    for depth in (0, 1, 4):
        a = g.trace_backward(ids, n_rays=20_000, max_depth=depth, keep_rejected=True).records()
        sa = dict(g.last_stats)
        b = g.trace_backward(ids, n_rays=20_000, max_depth=depth, keep_rejected=True,
                             breadth_first=True).records()
        assert np.array_equal(a, b) and sa["segments"] == g.last_stats["segments"]
        assert sa["candidates"] == g.last_stats["candidates"]
