"""Calls of different sizes from two host threads at once (ctypes releases the
interpreter lock): per-frame trees and channel correlations whose kernels take
different amounts of shared memory.  Every call succeeds and gives what it
gives alone."""
import dataclasses
import threading

import numpy as np
import pytest

from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _together(jobs):
    failed = []
    start = threading.Barrier(len(jobs))

    def run(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(4000):
                    job()
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # noqa: BLE001 - reported by the assertion below
            failed.append(repr(e))

    ts = [threading.Thread(target=run, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not failed, failed


def test_two_scenes_updated_at_once():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    jobs, made = [], []
    for n in (14_000, 30_000):
        rng = np.random.default_rng(n)
        sc = S.toy_scene(seed=0)
        rx = np.column_stack([rng.uniform(-90, 90, (n, 2)), rng.uniform(1, 3, n)]).astype(np.float32)
        fr = dataclasses.replace(sc.frame(0), rx_pos=rx, rx_vel=np.zeros_like(rx))
        fr = dataclasses.replace(fr, **{k: torch.as_tensor(getattr(fr, k)).cuda() for k in
                                        ("veh_pos", "veh_vel", "rx_pos", "rx_vel", "tx_pos", "tx_vel")})
        g = engine.Scene(sc, max_rx=n)
        g.update(fr)
        made.append((g, g.trace(n_rays=20_000).records()))
        jobs.append(lambda g=g, fr=fr: g.update(fr))
    torch.cuda.synchronize()
    _together(jobs)
    torch.cuda.synchronize()
    for g, want in made:
        assert len(want) and np.array_equal(g.trace(n_rays=20_000).records(), want)


def test_two_correlations_at_once():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    jobs, made = [], []
    for frames in (800, 1500):
        h = torch.rand((frames, 9, 2), generator=torch.Generator().manual_seed(frames),
                       dtype=torch.float64).cuda()
        made.append((h, engine.channel_correlation(h, 3)))
        jobs.append(lambda h=h: engine.channel_correlation(h, 3))
    torch.cuda.synchronize()
    _together(jobs)
    for h, want in made:
        assert torch.equal(engine.channel_correlation(h, 3), want)
