"""Backward discovery from a source list that holds receiver ids past the
present frame's (kept from a frame with more receivers, up to and beyond the
scene's capacity): they give no path, and the others' paths are those of the
list without them."""
import dataclasses

import numpy as np
import pytest

from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stale", [[10], [10, 11, 25, 39], [40], [1000, 2 ** 31 - 1]])
def test_ids_past_the_frame(stale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    sc = S.toy_scene(seed=2)
    rng = np.random.default_rng(5)
    rx = np.column_stack([rng.uniform(-60, 60, (40, 2)), rng.uniform(1, 3, 40)]).astype(np.float32)
    tx = np.float32([[-10, 4, 20], [15, -8, 25], [2, 3, 30]])
    fr = dataclasses.replace(sc.frame(0), rx_pos=rx, rx_vel=np.zeros_like(rx), tx_pos=tx,
                             tx_vel=np.zeros_like(tx))
    few = dataclasses.replace(fr, rx_pos=rx[:10], rx_vel=np.zeros_like(rx[:10]))
    g = engine.Scene(sc, max_rx=40, max_tx=3)
    g.update(fr)
    g.update(few)
    good = [0, 9, 4]

    def paths(ids):
        return g.trace_backward(torch.tensor(ids, dtype=torch.int32, device="cuda"),
                                n_rays=20_000).records()

    want = paths(good)
    assert set(want[:, 1].tolist()) == set(good) and set(want[:, 0].tolist()) == {0, 1, 2}
    assert np.array_equal(paths(good[:1] + stale + good[1:]), want)
