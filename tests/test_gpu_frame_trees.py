"""Per-frame trees built together (ranks by counting, boxes from aligned
blocks): the paths of a scene at sizes around a tile (512 keys), a block of
leaves (1024), a chunk and the largest size, against the breadth-first
receiver and vehicle queries of the other builders: every query is exact, so
the records are those of a scene object whose capacity takes it to the other
builders (frames above 32768 primitives).  Clustered positions share Morton
codes, so ties by index decide the order."""
import dataclasses

import numpy as np
import pytest

from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
MOST = 32768


def _frame(sc, n_rx, clustered, rng):
    fr = sc.frame(0)
    rx = np.column_stack([rng.uniform(-90, 90, n_rx), rng.uniform(-90, 90, n_rx),
                          rng.uniform(1.0, 3.0, n_rx)]).astype(np.float32)
    if clustered:
        h = n_rx // 2
        rx[:h] = (np.array([12.0, -7.0, 1.5]) + rng.uniform(0, 0.5, (h, 3))).astype(np.float32)
    return dataclasses.replace(fr, rx_pos=rx, rx_vel=np.zeros_like(rx))


def _with_vehicles(sc, n, rng):
    """The toy scene with n vehicle boxes on the ground."""
    pos = np.column_stack([rng.uniform(-90, 90, n), rng.uniform(-90, 90, n),
                           np.full(n, 0.75)]).astype(np.float32)
    half = np.tile(np.float32([[2.25, 0.9, 0.75]]), (n, 1))
    fr = dataclasses.replace(sc.frame(0), veh_pos=pos, veh_vel=np.zeros_like(pos))
    return dataclasses.replace(sc, veh_half=half, static_frame=fr)


@pytest.mark.parametrize("n_veh,n_rx,clustered", [
    (0, 1, False), (0, 2, False), (1, 1, False), (2, 3, False), (3, 512, False),
    (511, 513, True), (512, 1024, False), (1025, 1023, True), (1025, 1024, False),
    (2, 2046, True), (130, 4000, True),
    (4097, 300, False), (20, MOST - 20, True)])
def test_same_paths_as_the_other_builders(n_veh, n_rx, clustered):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    rng = np.random.default_rng(n_veh + n_rx)
    sc = _with_vehicles(S.toy_scene(seed=0), n_veh, rng)
    fr = _frame(sc, n_rx, clustered, rng)
    small = dataclasses.replace(sc, static_frame=fr)
    g = engine.Scene(small)
    g.update(fr)
    rec = g.trace(n_rays=30_000).records()
    seg = list(g.last_stats["segments"])
    # the same receivers with enough others, far above the scene, for the
    # other builders
    extra = MOST + 1 - n_veh - n_rx if n_veh + n_rx <= MOST else 0
    far = np.column_stack([rng.uniform(-90, 90, extra), rng.uniform(-90, 90, extra),
                           np.full(extra, 900.0)]).astype(np.float32)
    rx = np.concatenate([fr.rx_pos, far])
    big = dataclasses.replace(fr, rx_pos=rx, rx_vel=np.zeros_like(rx))
    h = engine.Scene(dataclasses.replace(sc, static_frame=big))
    h.update(big)
    want = h.trace(n_rays=30_000).records()
    want = want[want[:, 1] < n_rx]
    assert np.array_equal(rec, want)
    assert seg == list(h.last_stats["segments"])
    # back to few receivers on the same object: the trees of this frame again
    h.update(fr)
    assert np.array_equal(h.trace(n_rays=30_000).records(), rec)


def test_refit_between_rebuilds_gives_the_same_paths():
    """rebuild_every > 1: the vehicle tree is refitted in between, the other
    two trees are built; the records do not depend on it."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    sc = S.district_scene(seed=2, n_rays=100_000)
    a, b = engine.Scene(sc), engine.Scene(sc, rebuild_every=3)
    for k in range(5):
        a.update(sc.frame(k))
        b.update(sc.frame(k))
        assert np.array_equal(a.trace().records(), b.trace().records())
