"""Scratch that grows inside a relaxed stream capture: the zeros of its table of
candidates already met are then only recorded, so the next call issues them
itself.  A trace between the capture and its replay, and one after it, give the
records of a scene without captures; a receiver at each transmitter makes lists
long enough to use the table."""
import dataclasses

import numpy as np
import pytest

from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["revalidate", "trace"])
def test_growth_in_a_capture(call):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    sc = S.toy_scene(seed=1)
    rng = np.random.default_rng(4)
    rx = np.column_stack([rng.uniform(-60, 60, (30, 2)), rng.uniform(1, 3, 30)]).astype(np.float32)
    tx = np.float32([[-10, 4, 20], [5, -8, 25]])
    rx[7], rx[29] = tx
    fr = dataclasses.replace(sc.frame(0), rx_pos=rx, rx_vel=np.zeros_like(rx), tx_pos=tx,
                             tx_vel=np.zeros_like(tx))
    sc = dataclasses.replace(sc, static_frame=fr)
    rays, room = 4000, 300_000
    h = engine.Scene(sc)
    h.update(fr)
    want = h.trace(n_rays=rays).records()
    assert h.last_stats["candidates"] > 2 * 256 and len(want)

    g = engine.Scene(sc)
    g.update(fr)
    g.trace(n_rays=rays)  # everything but the larger scratch
    p = engine.Paths(room, g.device)
    p.rec[:len(want)] = torch.from_numpy(want.view(np.int32)).cuda()
    p.count.fill_(len(want))
    dirty = torch.full((room * 64,), 0x01010101, dtype=torch.int32, device="cuda")
    del dirty  # the capture gives it back to the device
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
        if call == "revalidate":
            g.revalidate(p)
        else:
            g.trace_async(p, n_rays=rays)
    for _ in range(2):
        assert np.array_equal(g.trace(n_rays=rays).records(), want)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(p.records(), want)
