"""Correlations of few pairs over many lags, whose lag passes (64 lags) are
shared among blocks: the same bits as each pass alone would give -- a
correlation to a smaller largest lag is a prefix, whatever the split -- at the
edges of a pass, in series held whole (to 1536 frames) and in chunks, against
plain torch within 200 F 2^-53 (F terms of magnitudes within a factor of a few,
over a variance of at least mu^2 / 50, both sides); and the time of many lags."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("frames,pairs,lag", [
    (100, 1, 63), (100, 1, 64), (130, 3, 128), (1536, 9, 700), (1537, 9, 700), (2500, 1, 2600),
    (300, 2500, 130), (5000, 17, 1000)])
def test_split_passes(frames, pairs, lag):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    gen = torch.Generator().manual_seed(frames + 31 * pairs + lag)
    h = (torch.rand(frames, pairs, 2, generator=gen, dtype=torch.float64) + 0.1).cuda()
    h[:, pairs // 2, :] *= 3.0
    R = engine.channel_correlation(h, lag)
    for less in (0, 62, 64, lag // 2):
        if less <= lag:
            assert torch.equal(R[:, :less + 1], engine.channel_correlation(h, less))
    R = R.cpu()
    g = h.cpu().square().sum(-1).sqrt()
    mu = g.mean(0)
    var = ((g - mu) ** 2).mean(0)
    assert bool((var > mu * mu / 50).all())
    for tau in range(0, lag + 1, 13):
        if tau >= frames:
            assert torch.all(R[:, tau] == 0)
            continue
        want = ((g[:frames - tau] * g[tau:]).mean(0) - mu * mu) / var
        assert torch.all((R[:, tau] - want).abs() <= 200 * frames * 2.0 ** -53)


def test_many_lags_of_one_pair_share_the_gpu():
    """24 passes cost no more than six times one (24 times in one block)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    h = torch.rand(4000, 1, 2, generator=torch.Generator().manual_seed(1), dtype=torch.float64).cuda()
    took = []
    for lag in (63, 24 * 64 - 1):
        best = 1e30
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            engine.channel_correlation(h, lag)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        took.append(best)
    assert took[1] < 6 * took[0], took
