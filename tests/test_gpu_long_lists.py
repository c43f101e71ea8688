"""Pairs with more candidates than are ordered by counting all against all
(256): a receiver exactly at a transmitter, which every primary ray meets, and
a ring of narrow mirrors that gives one pair hundreds of paths.  Records, and the
smallest ray index of each, equal the union of the same rays traced in parts
whose lists stay short; the work of the first grows with the rays, not with
their square."""
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


def _at_transmitter(n_rx=30):
    sc = S.toy_scene(seed=1)
    rng = np.random.default_rng(4)
    rx = np.column_stack([rng.uniform(-60, 60, (n_rx, 2)), rng.uniform(1, 3, n_rx)]).astype(np.float32)
    tx = np.float32([[-10, 4, 20], [5, -8, 25]])
    rx[7], rx[n_rx - 1] = tx[0], tx[1]
    fr = dataclasses.replace(sc.frame(0), rx_pos=rx, rx_vel=np.zeros_like(rx), tx_pos=tx,
                             tx_vel=np.zeros_like(tx))
    return dataclasses.replace(sc, static_frame=fr), fr


def _mirrors():
    n, r = 1200, 20.0
    a = 2 * np.pi * np.arange(n + 1) / n
    polys = []
    for k in range(n):  # facing the centre
        x0, y0, x1, y1 = (r * np.cos(a[k]), r * np.sin(a[k]), r * np.cos(a[k + 1]), r * np.sin(a[k + 1]))
        polys.append([(x1, y1, 0), (x0, y0, 0), (x0, y0, 6), (x1, y1, 6)])
    sc = S.custom_scene(polys, [2] * n, [(0.0, 0.0, 3.0)], [(0.003, 0.002, 3.1), (4.0, 1.0, 2.0)], depth=1)
    return sc, sc.frame(0)


def _rows(rec):
    d = rec[:, 2] & 15
    f = np.where(np.arange(4) < d[:, None], rec[:, 3:7], 0)
    return np.column_stack([rec[:, 0], rec[:, 1], d, f]).astype(np.int64)


@pytest.mark.parametrize("which,n_rays,parts", [
    ("transmitter", 255, 1), ("transmitter", 256, 2), ("transmitter", 257, 2),
    ("transmitter", 4000, 40), ("mirrors", 100_000, 40)])
def test_long_lists_equal_short_ones(engine, which, n_rays, parts):
    sc, fr = _at_transmitter() if which == "transmitter" else _mirrors()
    g = engine.Scene(sc)
    g.update(fr)
    best, cand = {}, 0
    for k in range(parts):
        rec = g.trace(n_rays=n_rays, offset=k, stride=parts, keep_rejected=True).records()
        cand += g.last_stats["candidates"]
        for row, j in zip(map(tuple, _rows(rec)), rec[:, 7].astype(np.int64) * parts + k):
            best[row] = min(best.get(row, 1 << 40), int(j))
    for _ in range(3):  # the table is empty again after each
        rec = g.trace(n_rays=n_rays, keep_rejected=True).records()
        assert g.last_stats["candidates"] == cand
        rows = list(map(tuple, _rows(rec)))
        assert rows == sorted(best) and g.last_stats["unique_candidates"] == len(rows)
        assert rec[:, 7].tolist() == [best[r] for r in rows]
    if which == "mirrors":
        assert (rec[:, 1] == 0).sum() > 2 * 256
    # in a batch beside an ordinary scene
    other, fo = S.toy_scene(seed=3), S.toy_scene(seed=3).frame(0)
    h = engine.Scene(other)
    h.update(fo)
    alone = h.trace(n_rays=5000).records()
    want = g.trace(n_rays=n_rays).records()
    b = engine.Batch([h, g, h], params=[dict(n_rays=5000), dict(n_rays=n_rays), dict(n_rays=5000)],
                     capacity=[20_000] * 3)
    for _ in range(2):
        b.trace_async()
        b.sync()
        for out, w in zip(b.outs, (alone, want, alone)):
            assert np.array_equal(out.records(), w)


def test_a_receiver_at_a_transmitter_costs_its_rays(engine):
    """A list ordered all against all would take 16 times as long with four
    times the rays."""
    sc, fr = _at_transmitter()
    g = engine.Scene(sc)
    g.update(fr)
    took = []
    for n in (50_000, 200_000):
        p = g.trace(n_rays=n, max_depth=0)
        assert g.last_stats["candidates"] >= 2 * n
        out = engine.Paths(p.capacity, g.device)
        best = 1e30
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            g.trace_async(out, n_rays=n, max_depth=0)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        took.append(best)
    assert took[1] < 8 * took[0], took
