"""Per-frame trees of frames whose primitives crowd into few Morton bins: crowds
of sizes around the length from which a bin is no longer compared all with all
(256) and around a block of 256 places, several in a row, of vehicles and
receivers together, and of equal positions.  Paths equal those of the builders
for frames above 32768 primitives; a crowd costs no more than three times a
spread frame."""
import dataclasses

import numpy as np
import pytest

from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
MOST = 32768
NAMES = ("veh_pos", "veh_vel", "rx_pos", "rx_vel", "tx_pos", "tx_vel")


def _crowds(sizes, spread, total, rng):
    """Points in crowds of these sizes, crowd k at its own place, the rest of
    total anywhere, in random order."""
    at = [np.array([15.0, -7.0, 1.5] if k == 0 else [-70 + 11.0 * (k % 13), -60 + 13.0 * (k // 13), 1.5])
          for k in range(len(sizes))]
    p = [c + (rng.uniform(0, spread, (n, 3)) if spread else np.zeros((n, 3))) for c, n in zip(at, sizes)]
    rest = total - sum(sizes)
    p.append(np.column_stack([rng.uniform(-90, 90, (rest, 2)), rng.uniform(1, 3, rest)]))
    return rng.permutation(np.concatenate(p)).astype(np.float32)


def _scene(n_veh, sizes, spread, total, seed):
    rng = np.random.default_rng(seed)
    sc = S.toy_scene(seed=0)
    fr = sc.frame(0)
    rx = _crowds(sizes, spread, total, rng)
    if n_veh:  # the vehicles crowd beside the first receivers
        pos = np.column_stack([rng.uniform(19, 22, (n_veh, 1)), rng.uniform(-7, -5, (n_veh, 1)),
                               np.full(n_veh, 0.75)]).astype(np.float32)
        half = np.tile(np.float32([[0.4, 0.3, 0.75]]), (n_veh, 1))
        fr = dataclasses.replace(fr, veh_pos=pos, veh_vel=np.zeros_like(pos))
        sc = dataclasses.replace(sc, veh_half=half)
    fr = dataclasses.replace(fr, rx_pos=rx, rx_vel=np.zeros_like(rx))
    return dataclasses.replace(sc, static_frame=fr), fr


@pytest.mark.parametrize("n_veh,sizes,spread,total", [
    (0, (255, 256, 257), 0.5, 1200), (0, (1000,), 0.5, 1500), (0, (2048,), 0.0, 2048), (0, (257,), 0.0, 257), (0, (256,), 0.0, 256), (0, (1025,), 0.0, 1100),
    (300, (500, 64, 257), 0.5, 1700), (600, (700, 700), 0.0, 1448),
    (0, (255, 256, 257, 258, 511, 512, 513), 0.5, 2600), (0, (300,) * 20, 0.5, 6000),
    (0, (2049,), 0.0, 2049), (900, (257, 300, 5000), 0.5, 9000), (1500, (4000,), 0.0, 5000),
    (3000, (20_000, 300, 290), 0.5, MOST - 3000), (0, (MOST,), 0.0, MOST)])
def test_crowds_give_the_paths_of_the_other_builders(n_veh, sizes, spread, total):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    sc, fr = _scene(n_veh, sizes, spread, total, n_veh + total)
    g = engine.Scene(sc)
    g.update(fr)
    rec = g.trace(n_rays=3_000, max_depth=1).records()
    seg = list(g.last_stats["segments"])
    extra = MOST + 1 - n_veh - total
    far = np.column_stack([np.random.default_rng(1).uniform(-90, 90, (extra, 2)), np.full(extra, 900.0)])
    rx = np.concatenate([fr.rx_pos, far.astype(np.float32)])
    big = dataclasses.replace(fr, rx_pos=rx, rx_vel=np.zeros_like(rx))
    h = engine.Scene(dataclasses.replace(sc, static_frame=big))
    h.update(big)
    want = h.trace(n_rays=3_000, max_depth=1).records()
    want = want[want[:, 1] < total]
    assert len(rec) >= min(total, 64) and np.array_equal(rec, want)
    assert seg == list(h.last_stats["segments"])


@pytest.mark.parametrize("total", [2000, 4000, 15_000, 32_700])
def test_a_crowd_costs_what_a_spread_frame_does(total):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    took = []
    for sizes, spread in (((), 0.0), ((total,), 0.5), ((total,), 0.0)):
        sc, fr = _scene(0, sizes, spread, total, total)
        fr = dataclasses.replace(fr, **{k: torch.as_tensor(getattr(fr, k)).cuda() for k in NAMES})
        g = engine.Scene(sc)
        best = 1e30
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(20):
                g.update(fr)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        took.append(best)
    assert max(took[1:]) < 3 * took[0], took
