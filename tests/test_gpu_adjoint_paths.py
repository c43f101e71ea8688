"""Adjoint of the field at the edges of its kernel (eight paths a warp, four
lanes a path): path counts around a warp, depths 0-4, vehicle faces, normal
incidence, constant-Gamma mode, against central differences of the oracle's
FP64 field for the linear loss sum(cot * h).

Tolerance, with A = sum over the paths of |a| |cot|: the amplitude's phase
turns by w = 2 pi f / c = 73.4 rad per metre of path length, and a step h in
the transmitter changes a length by at most h, so a difference of step h has
truncation (w h)^2 / 6 of w A, 9e-6 at h = 1e-4 m (at most doubled by the
float32 step's rounding up); rounding, 1e-16 x 1e4 rad over w h = 7e-3, is
1e-10.  Allowed: 1e-4 w A.  A relative change of a material parameter by
1e-4 gives truncation 1e-8 times derivatives of the Fresnel coefficients of
order one per bounce; allowed: 1e-5 x 4 A per relative change."""
import dataclasses

import numpy as np
import pytest

import oracle
from helpers import rec_to_paths
from paper_2303_10521_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _canyon(n_rx, seed):
    rng = np.random.default_rng(seed)
    polys = [S.rect_xy(-40, -40, 40, 40), S.rect_wall_x(12.0, -40, 40, 0, 30),
             S.rect_wall_x(-9.0, -40, 40, 0, 30, facing=1)]
    rx = np.stack([rng.uniform(-8, 11, n_rx), rng.uniform(-15, 15, n_rx),
                   rng.uniform(1, 6, n_rx)], 1)
    # receiver 0 straight across from transmitter 0: normal incidence on the walls
    rx[0] = (5.0, -3.0, 9.0)
    return S.custom_scene(polys, [0, 2, 3], [(1.5, -3.0, 9.0), (-2.0, 6.0, 7.5)], rx,
                          boxes=[((3, -2, 0.25), (5, 3, 1.75))], n_rays=200_000, depth=4)


@pytest.fixture(scope="module")
def canyon():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_10521_gb300 import engine
    sc = _canyon(24, 3)
    g = engine.Scene(sc)
    g.update(sc.frame(0))
    return engine, sc, g, g.trace().records()


@pytest.mark.parametrize("n,const_gamma", [(1, False), (7, False), (8, False), (9, False),
                                           (33, False), (33, True), (None, False)])
def test_adjoint_matches_differences(canyon, n, const_gamma):
    engine, sc, g, rec = canyon
    depths = set((rec[:, 2] & 15).tolist())
    assert depths == {0, 1, 2, 3, 4} and (rec[:, 3:7].min(1) < 3).any()
    if n is not None:  # a subset of n paths of every depth, in canonical order
        pick = np.sort(np.random.default_rng(n).permutation(len(rec))[:n])
        rec = rec[pick]
    n = len(rec)
    p = engine.Paths(n, "cuda")
    p.rec[:] = torch.from_numpy(rec.view(np.int32)).cuda()
    p.count.fill_(n)
    fr, f, po = sc.frame(0), sc.freqs[0], rec_to_paths(rec)
    cot = np.random.default_rng(7).normal(size=(2, 24, 2))
    c = cot[po["tx"], po["rx"]]

    def loss(frame, eps, sig):
        o = oracle.OracleScene(sc, frame, const_gamma, eps_r=eps, sigma=sig)
        a, _, _ = oracle.field(o, po, f)
        return float((c[:, 0] * a.real + c[:, 1] * a.imag).sum())

    a0, _, _ = oracle.field(oracle.OracleScene(sc, fr, const_gamma), po, f)
    A = float((np.abs(a0) * np.linalg.norm(c, axis=1)).sum())
    ge, gs, gt = (t.cpu().numpy() for t in g.channel_backward(
        p, f, torch.as_tensor(cot).cuda(), const_gamma=const_gamma))
    for got, base, which in ((ge, sc.eps_r, 0), (gs, sc.sigma, 1)):
        for m in range(8):
            v = []
            for s in (1.0, -1.0):
                q = base.copy()
                q[m] *= 1.0 + s * 1e-4
                v.append(loss(fr, *((q, sc.sigma) if which == 0 else (sc.eps_r, q))))
            want = (v[0] - v[1]) / 2e-4
            assert abs(got[m] * base[m] - want) <= 1e-5 * 4 * A
    for t in range(2):
        for k in range(3):
            x = float(fr.tx_pos[t, k])
            h = 2.0 ** -13  # exact in float32 at these positions
            v = []
            for s in (h, -h):
                q = fr.tx_pos.copy()
                q[t, k] = np.float32(x + s)
                assert float(q[t, k]) == x + s
                v.append(loss(dataclasses.replace(fr, tx_pos=q), sc.eps_r, sc.sigma))
            assert abs(gt[t, k] - (v[0] - v[1]) / (2 * h)) <= 1e-4 * 73.4 * A
