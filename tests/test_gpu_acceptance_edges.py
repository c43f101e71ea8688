"""Acceptance with the FP32-first face margin and occlusion legs in pieces:
records whose reflection points lie on, just inside and just outside face
edges (walls, a 14-gon roof, a 2 km ground, at 1 km from the origin), and legs of
lengths around a piece and the largest piece count, against the oracle's FP64
acceptance.  A verdict may differ only where the oracle flags the path as
within 1e-4 m of a boundary (whole numbers otherwise equal); the GPU's own
margin flag equals the FP64 margin test of the same points."""
import numpy as np
import pytest

import oracle
from helpers import rec_to_paths
from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _revalidated(engine, sc, rec):
    g = engine.Scene(sc)
    g.update(sc.frame(0))
    p = engine.Paths(len(rec), g.device)
    p.rec[:] = torch.from_numpy(rec.view(np.int32)).cuda()
    p.count.fill_(len(rec))
    g.revalidate(p, keep=True)
    g.sync()
    return p.records()


def _record(tx, rx, faces):
    k = len(faces)
    return [tx, rx, k] + faces + [0xffffffff] * (4 - k) + [0]


@pytest.mark.parametrize("origin", [0.0, 1000.0])
def test_reflection_points_at_face_edges(origin):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    ang = 2 * np.pi * np.arange(14) / 14
    roof = [(origin + 8 * np.cos(t), 8 * np.sin(t), 12.0) for t in ang]
    polys = [S.rect_xy(-1000, -1000, 1000, 1000), roof,
             S.rect_wall_x(origin + 30.0, -6, 6, 13, 25)]
    # single reflections off the roof (z = 12) and the wall (x = origin + 30)
    # between points at equal heights / distances, so that the reflection point
    # is the midpoint: put it at signed distances from edges and corners
    tx = np.float32([[origin + 0.0, 0.0, 16.0]])
    pts = []
    for d in (0.0, 1e-6, 3e-5, 9e-5, 1.1e-4, 1e-3, 0.05, 1.0):
        for s in (-1.0, 1.0):
            for t in (0.0, ang[1] / 2, 0.3):
                r = (8 * np.cos(np.pi / 14) if t else 8.0) + s * d
                pts.append((2 * r * np.cos(t), 2 * r * np.sin(t), 16.0, [1]))
            pts.append((0.0, 2 * (6 + s * d), 16.0, [2]))
            pts.append((3.0, 1.0, 2 * (13 + s * d) - 16.0, [2]))
            pts.append((2 * d, -40.0, 16.0, [0]))
    rx = np.float32([[origin + x, y, z] for x, y, z, _ in pts])
    sc = S.custom_scene(polys, [0, 2, 3], tx, rx)
    rec = np.array([_record(0, i, p[3]) for i, p in enumerate(pts)], np.uint32)
    got = _revalidated(engine, sc, rec)
    o = oracle.OracleScene(sc, sc.frame(0))
    want, marg = oracle.validate(o, rec_to_paths(rec))
    ok = (got[:, 2] & 0x100) != 0
    marg = np.asarray(marg) != 0
    assert np.array_equal(ok[~marg], np.asarray(want, bool)[~marg])
    assert ok.any() and (~ok).any() and marg.any() and (~marg).any()
    # a path the GPU calls marginal is one the oracle does
    assert np.all(marg[(got[:, 2] & 0x200) != 0])


@pytest.mark.parametrize("n", [1, 7, 40, 700])
def test_legs_of_every_length(n):
    """Lines of sight of 1 m to 1.9 km over a row of thin walls with gaps."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    rng = np.random.default_rng(n)
    polys = [S.rect_xy(-1000, -1000, 1000, 1000)]
    for k in range(37):
        polys.append(S.rect_wall_x(-900.0 + 50 * k, -400 + 11 * k, 400 - 7 * k, 0, 8 + (k % 5)))
    d = np.exp(rng.uniform(0, np.log(1900), n))
    d[:min(n, 6)] = (63.9, 64.0, 64.1, 256.0, 1023.0, 1100.0)[:min(n, 6)]
    rx = np.column_stack([-950 + d, rng.uniform(-3, 3, n), rng.uniform(1, 30, n)]).astype(np.float32)
    sc = S.custom_scene(polys, [0] + [2] * 37, [(-950.0, 0.0, 9.0)], rx,
                        boxes=[((-600, -2, 5), (-596, 2, 9))])
    rec = np.array([_record(0, i, []) for i in range(n)], np.uint32)
    got = _revalidated(engine, sc, rec)
    want, marg = oracle.validate(oracle.OracleScene(sc, sc.frame(0)), rec_to_paths(rec))
    marg = np.asarray(marg) != 0
    assert np.array_equal(((got[:, 2] & 0x100) != 0)[~marg], np.asarray(want, bool)[~marg])
    assert (~marg).sum() >= 0.8 * n
