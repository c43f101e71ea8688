"""Eq. 1 correlation at the edges of its kernel: pairs around a block's 8,
lags around a lag group (4), a warp (16) and a pass (64), lags beyond the
series, one frame, and series longer than shared memory holds (chunked form),
against plain torch in 64 bits.  The sums have F terms of magnitudes within a
factor of a few of one another, so mean and covariance carry at most F 2^-53
relative error; divided by a variance of at least mu^2 / 50 and doubled for
the two sides, |dR| <= 200 F 2^-53."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("frames,pairs,lag", [
    (1, 1, 0), (1, 3, 5), (2, 7, 1), (17, 8, 16), (40, 9, 15), (64, 33, 63), (70, 5, 64),
    (65, 31, 200), (300, 100, 50), (1536, 9, 17), (1537, 9, 70), (2600, 3, 130)])
def test_correlation_sizes(frames, pairs, lag):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    gen = torch.Generator().manual_seed(frames + 31 * pairs + lag)
    # an offset of one double: the series need not be 16-byte aligned
    flat = torch.rand(frames * pairs * 2 + 1, generator=gen, dtype=torch.float64) + 0.1
    h = flat.cuda()[1:].view(frames, pairs, 2)
    if frames > 2:
        h[:, 0] = 0.0  # a pair without paths: R = 0
    R = engine.channel_correlation(h, lag).cpu()
    g = h.cpu().square().sum(-1).sqrt()
    mu = g.mean(0)
    var = ((g - mu) ** 2).mean(0)
    assert R.shape == (pairs, lag + 1)
    for tau in range(lag + 1):
        if tau >= frames:
            assert torch.all(R[:, tau] == 0)
            continue
        want = ((g[:frames - tau] * g[tau:]).mean(0) - mu * mu)
        live = var > mu * mu / 50
        if frames > 2:
            assert not live[0] and R[0, tau] == 0
        assert torch.all((R[:, tau] - want / var)[live].abs() <= 200 * frames * 2.0 ** -53)
