"""Acceptance at the sides of large slanted faces with a short, nearly
collinear edge far from the face's first vertex: reflection points within 2 m of the
side that the short edge continues.  The verdict equals the FP64 margin's, and
so does the margin flag, wherever the FP64 margin (formed here in numpy from
the same float32 inputs, its own rounding below 1e-9 m) is not within 1e-9 m of
a threshold."""
import numpy as np
import pytest

from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
Z, H = 0.0, 30.0


def _face(length, width, short, rng):
    """A rotated rectangle off the origin, one vertex more at `short` from the
    end of its first side, convex after rounding to float32; the first side's
    ends; the vertex order starts away from the short edge."""
    while True:
        th = rng.uniform(0, 2 * np.pi)
        rot = np.array([[np.cos(th), -np.sin(th)], [np.sin(th), np.cos(th)]])
        q = np.array([[-length, -width], [length - 2 * short, -width - rng.uniform(0, 6e-5)],
                      [length, -width], [length, width], [-length, width]]) / 2
        v = (q @ rot.T + rng.uniform(-500, 500, 2)).astype(np.float32)
        e = np.roll(v, -1, 0).astype(np.float64) - v
        n = np.roll(e, -1, 0)
        if (e[:, 0] * n[:, 1] - e[:, 1] * n[:, 0]).min() > 0:
            return np.roll(v, rng.integers(1, 4), 0), v[0].astype(float), v[2].astype(float)


def _margin(v, p):
    a, b = np.roll(v, 1, 0).astype(np.float64), v.astype(np.float64)
    e, w = b - a, p[:, None, :] - a[None]
    return ((e[:, 0] * w[..., 1] - e[:, 1] * w[..., 0]) / np.hypot(e[:, 0], e[:, 1])).min(1)


@pytest.mark.parametrize("length,width,short", [
    (1000, 800, 0.02), (1000, 800, 0.1), (1000, 800, 2.0), (2000, 1600, 2.6), (60, 20, 0.02)])
def test_sides_with_a_short_edge(length, width, short):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    rng = np.random.default_rng(int(1000 * short) + length)
    both = np.zeros(2, bool)
    for _ in range(12):
        v, s0, s1 = _face(length, width, short, rng)
        side = (s1 - s0) / np.hypot(*(s1 - s0))
        inward = np.array([-side[1], side[0]])
        n = 3000
        d = rng.choice([-2.0, 2.0], n) * np.exp(rng.uniform(np.log(1e-5), 0, n))
        at = s0 + rng.uniform(0.02, 0.98, n)[:, None] * (s1 - s0) + d[:, None] * inward
        # transmitter and receivers at one height: reflected half way
        tx = v.mean(0).astype(np.float64)
        rx = np.column_stack([2 * at - tx, np.full(n, H)]).astype(np.float32)
        txf = np.float32([tx[0], tx[1], H])
        sc = S.custom_scene([np.column_stack([v, np.full(5, Z)])], [0], txf, rx)
        rec = np.full((n, 8), 0xffffffff, np.uint32)
        rec[:, 0], rec[:, 1], rec[:, 2], rec[:, 3], rec[:, 7] = 0, np.arange(n), 1, 0, 0
        g = engine.Scene(sc)
        g.update(sc.frame(0))
        p = engine.Paths(n, g.device)
        p.rec[:] = torch.from_numpy(rec.view(np.int32)).cuda()
        p.count.fill_(n)
        g.revalidate(p, keep=True)
        g.sync()
        got = p.records()[:, 2]
        m = _margin(v, (rx[:, :2].astype(np.float64) + txf[:2].astype(np.float64)) / 2)
        sure = np.abs(m) > 1e-9
        assert np.array_equal(((got & 0x100) != 0)[sure], (m >= 0)[sure])
        sure = np.abs(np.abs(m) - 1e-4) > 1e-9
        assert np.array_equal(((got & 0x200) != 0)[sure], (np.abs(m) < 1e-4)[sure])
        both |= np.array([(m > 1e-4).any(), (m < -1e-4).any()])
    assert both.all()
