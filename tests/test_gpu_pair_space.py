"""The per-pair counts of a trace have a fixed size: a trace captured into a
graph may have more receivers than any trace before it, and a batch whose
receiver capacities make more than 2^20 pairs lists neighbouring receivers
together.  Records equal those of the same traces issued one by one."""
import dataclasses

import numpy as np
import pytest

from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
NAMES = ("veh_pos", "veh_vel", "rx_pos", "rx_vel", "tx_pos", "tx_vel")


@pytest.fixture(scope="module")
def engine():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine as E
    return E


def _frame(sc, n_rx, n_tx, seed):
    rng = np.random.default_rng(seed)
    rx = np.column_stack([rng.uniform(-80, 80, (n_rx, 2)), rng.uniform(1, 3, n_rx)]).astype(np.float32)
    tx = np.column_stack([rng.uniform(-20, 20, (n_tx, 2)), rng.uniform(8, 40, n_tx)]).astype(np.float32)
    return dataclasses.replace(sc.frame(0), rx_pos=rx, rx_vel=np.zeros_like(rx), tx_pos=tx,
                               tx_vel=np.zeros_like(tx))


def test_captured_trace_with_more_receivers_than_before(engine):
    sc = S.toy_scene(seed=0)
    g = engine.Scene(sc, max_rx=700, max_tx=2)
    few, many = _frame(sc, 5, 2, 1), _frame(sc, 700, 2, 2)
    many = dataclasses.replace(many, **{k: torch.as_tensor(getattr(many, k)).cuda() for k in NAMES})
    kw = dict(n_rays=20_000, max_depth=2)
    out = engine.Paths(60_000, g.device)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        g.update(few)
        g.trace_async(out, **kw)  # sizes what the sizes of this call need
        g.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            g.update(many)
            g.trace_async(out, **kw)
        graph.replay()
        g.sync()
    got = out.records()
    h = engine.Scene(sc, max_rx=700, max_tx=2)
    h.update(many)
    want = h.trace(**kw).records()
    assert len(want) > 700 and np.array_equal(got, want)


@pytest.mark.parametrize("max_rx", [174_000, 300_001, 700_000])
def test_batch_of_many_possible_pairs(engine, max_rx):
    """3 scenes x 2 transmitters: below 2^20 pairs, 2 and 8 receivers a list."""
    scs = [S.toy_scene(seed=k) for k in range(3)]
    frs = [_frame(s, 900 + 7 * k, 2, 5 + k) for k, s in enumerate(scs)]
    scenes = []
    for s, f in zip(scs, frs):
        g = engine.Scene(s, max_rx=max_rx, max_tx=2)
        g.update(f)
        scenes.append(g)
    want = [g.trace(n_rays=20_000, max_depth=2).records() for g in scenes]
    b = engine.Batch(scenes, params=[dict(n_rays=20_000, max_depth=2)] * 3, capacity=[30_000] * 3)
    b.trace_async()
    b.sync()
    for p, w in zip(b.outs, want):
        assert len(w) > 900 and np.array_equal(p.records(), w)
