"""Candidates to canonical records (counted per pair, ordered within the
pair): the output against the same trace's candidates deduplicated on the host,
at sizes where the steps can go wrong -- one pair, pairs around a group of 256
and beyond, a pair holding hundreds of candidates, capacities that cut the
candidates or the records -- and the merge of a rediscovery against the set
union of the cache and the new paths.  Whole numbers: equal."""
import dataclasses

import numpy as np
import pytest

import oracle
from helpers import rec_to_paths
from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def engine():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine as E
    return E


def _scene(n_rx, n_tx, clustered=False):
    rng = np.random.default_rng([n_rx, n_tx])
    sc = S.toy_scene(seed=1)
    fr = sc.frame(0)
    xy = rng.uniform(-1, 1, (n_rx, 2)) if clustered else rng.uniform(-90, 90, (n_rx, 2))
    rx = np.column_stack([xy, rng.uniform(1, 3, n_rx)]).astype(np.float32)
    tx = np.column_stack([rng.uniform(-20, 20, (n_tx, 2)),
                          rng.uniform(8, 40, n_tx)]).astype(np.float32)
    fr = dataclasses.replace(fr, rx_pos=rx, rx_vel=np.zeros_like(rx), tx_pos=tx,
                             tx_vel=np.zeros_like(tx))
    return dataclasses.replace(sc, static_frame=fr), fr


def _words(rec):
    """Records without flags, as rows that sort in canonical order."""
    r = rec.astype(np.int64)
    d = r[:, 2] & 15
    f = np.where(np.arange(4) < d[:, None], r[:, 3:7], 0)
    return np.column_stack([r[:, 0], r[:, 1], d, f])


@pytest.mark.parametrize("n_rx,n_tx,n_rays,depth", [
    (1, 1, 60_000, 4), (255, 1, 20_000, 3), (256, 2, 20_000, 2), (1025, 1, 20_000, 2),
    (2000, 3, 5_000, 4)])
def test_records_are_the_candidates_in_canonical_order(engine, n_rx, n_tx, n_rays, depth):
    """The same rays in two halves, each traced alone: the whole trace holds
    the union of their paths with the smaller ray index, ordered."""
    sc, fr = _scene(n_rx, n_tx)
    g = engine.Scene(sc)
    g.update(fr)
    whole = g.trace(n_rays=n_rays, max_depth=depth, keep_rejected=True).records()
    st = dict(g.last_stats)
    n0 = (n_rays + 1) // 2
    a = g.trace(n_rays=n_rays, max_depth=depth, offset=0, stride=2, keep_rejected=True).records()
    ca = g.last_stats["candidates"]
    b = g.trace(n_rays=n_rays, max_depth=depth, offset=1, stride=2, keep_rejected=True).records()
    assert ca + g.last_stats["candidates"] == st["candidates"] and n0 > 0
    w = _words(whole)
    assert st["unique_candidates"] == len(w) > 0
    assert np.array_equal(w, np.unique(w, axis=0))  # ordered, no duplicates
    both = np.concatenate([_words(a), _words(b)])
    assert np.array_equal(w, np.unique(both, axis=0))
    ray = {}
    for rows, rec, off in ((_words(a), a, 0), (_words(b), b, 1)):
        for k, j in zip(map(tuple, rows), rec[:, 7].astype(np.int64) * 2 + off):
            ray[k] = min(ray.get(k, 1 << 40), int(j))
    assert [ray[tuple(k)] for k in w] == whole[:, 7].tolist()
    kept = g.trace(n_rays=n_rays, max_depth=depth).records()
    valid = whole[(whole[:, 2] & 0x100) != 0]
    assert np.array_equal(kept, valid)


def test_more_pairs_than_one_scan_takes(engine):
    """16 x 70000 pairs (above 2^20: scanned by the general scan) against each
    of two transmitters traced alone (70000 pairs)."""
    sc, fr = _scene(70_000, 16)
    g = engine.Scene(sc)
    g.update(fr)
    kw = dict(n_rays=20_000, max_depth=0)
    whole = g.trace(**kw).records()
    assert len(whole) > 1000
    for t in (0, 11):
        one = dataclasses.replace(fr, tx_pos=fr.tx_pos[t:t + 1], tx_vel=fr.tx_vel[t:t + 1])
        g.update(one)
        alone = g.trace(**kw).records()
        part = whole[whole[:, 0] == t].copy()
        part[:, 0] = 0
        assert len(alone) > 100 and np.array_equal(alone, part)


def test_a_pair_with_many_candidates(engine):
    """40 receivers in one place and few, wide rays: pairs of hundreds of
    candidates of many paths; the oracle's deduplication of the same records."""
    sc, fr = _scene(40, 1, clustered=True)
    g = engine.Scene(sc)
    g.update(fr)
    rec = g.trace(n_rays=3_000_000, max_depth=4, count=3_000_000, keep_rejected=True).records()
    w = _words(rec)
    assert np.array_equal(w, np.unique(w, axis=0))
    per = np.bincount(rec[:, 1].astype(np.int64))
    assert per.max() >= 20
    p = rec_to_paths(rec)
    assert len(oracle.dedup(p)) == len(p)


def test_capacities(engine):
    sc, fr = _scene(300, 2)
    g = engine.Scene(sc)
    g.update(fr)
    full = g.trace(n_rays=30_000).records()
    cut = engine.Paths(len(full) - 5, g.device)
    g.trace_async(cut, n_rays=30_000)
    with pytest.raises(engine.N.EmrtError) as ei:
        g.sync()
    assert ei.value.code == 4 and cut.n() == len(full)
    assert np.array_equal(cut.records(), full[:len(full) - 5])


@pytest.mark.parametrize("revalidate", [False, True])
@pytest.mark.parametrize("kept", [0, 1, 2, 3])
def test_rediscovery_is_the_union(engine, revalidate, kept):
    """A cache of every kept-th path of a coarse trace (0: an empty cache) and
    a finer rediscovery."""
    sc, fr = _scene(700, 2)
    g = engine.Scene(sc)
    g.update(fr)
    coarse = g.trace(n_rays=9_000).records()
    fine = g.trace(n_rays=30_000).records()
    old = coarse[::kept] if kept else coarse[:0]
    cache = engine.Paths(len(coarse) + len(fine), g.device)
    if len(old):
        cache.rec[:len(old)] = torch.from_numpy(old.view(np.int32)).cuda()
    cache.count.fill_(len(old))
    g.rediscover(cache, n_rays=30_000, revalidate=revalidate)
    g.sync()
    got = cache.records()
    rows = np.unique(np.concatenate([_words(old), _words(fine)]), axis=0)
    assert np.array_equal(_words(got), rows)
    ray = {tuple(k): int(j) for k, j in zip(_words(old), old[:, 7])}
    for k, j in zip(map(tuple, _words(fine)), fine[:, 7]):
        ray[k] = min(ray.get(k, 1 << 40), int(j))
    assert [ray[tuple(k)] for k in rows] == got[:, 7].tolist()
    assert np.all(got[:, 2] & 0x100)
    # too little room: the count required, the first records, an error
    small = engine.Paths(len(rows) - 3, g.device)
    if len(old) <= small.capacity:
        small.rec[:len(old)] = torch.from_numpy(old.view(np.int32)).cuda()
        small.count.fill_(len(old))
        g.rediscover(small, n_rays=30_000, revalidate=revalidate)
        with pytest.raises(engine.N.EmrtError) as ei:
            g.sync()
        assert ei.value.code == 4 and small.n() == len(rows)
        assert np.array_equal(_words(small.records()), rows[:len(rows) - 3])
