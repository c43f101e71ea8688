"""The depth-first walk with many receivers and many rays, on both sides of the
rule that lets it ask for possible receivers before a last segment's end (n_rx
times the reception radius factor up to 2.5, or up to 10 from 2^24 rays):
records, segments and candidates equal the breadth-first form's, which always
looks for the end.  Each case states the side it takes."""
import numpy as np
import pytest

from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rx,n_rays,asks", [
    (4000, 9_000_000, True), (10_000, 9_000_000, True), (12_000, 9_000_000, False),
    (4000, 8_000_000, False), (2500, 9_000_000, True)])
def test_many_receivers_and_rays(n_rx, n_rays, asks):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    sc = S.district_scene(seed=3, n_veh=37, n_rx=n_rx, depth=2)
    fr = sc.frame(5)
    g = engine.Scene(sc)
    g.update(fr)
    met = n_rx * 1.25 * np.sqrt(8 * np.pi / (3 * np.sqrt(3) * n_rays))
    assert asks == (met <= 2.5 or (met <= 10 and n_rays * len(fr.tx_pos) >= 2 ** 24))
    a = g.trace(n_rays=n_rays, max_depth=2, keep_rejected=True).records()
    sa = dict(g.last_stats)
    b = g.trace(n_rays=n_rays, max_depth=2, keep_rejected=True, breadth_first=True).records()
    assert len(a) > n_rx and np.array_equal(a, b)
    assert sa["segments"] == g.last_stats["segments"]
    assert sa["candidates"] == g.last_stats["candidates"]
