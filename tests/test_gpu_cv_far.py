"""The quadratures against the FP64 ones where their tiling can go wrong: an odd
last triangle, one triangle, one either side of a tile, other point counts than
whole blocks, every subdivision level's fine nodes.

Bar: the terms' worst-case rounding.  With u = 2^-24 a term w (r . n)
(f - f_x) / (4 pi r^3) has a plane product off by at most 6 u (|r| + 2 |y|)
(node, normal, offset, four operations) and r^-3 by 12 u (the node's rounding
and six operations, times 3/2), so the sum by 24 u sum w (|r| + 2 |y|)
|f - f_x| / (4 pi r^3); a sum of m terms in FP32 adds at most 8 u of it.
"""
import numpy as np
import pytest

from oracle import cv as C
from paper_2305_04403_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tris,level,points", [(1280, 2, 300), (1279, 1, 33), (257, 1, 257), (256, 0, 1),
                                               (65, 3, 31), (63, 0, 129), (1, 2, 40)])
def test_quadrature_tiles(tris, level, points):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_04403_gb300 as wob
    v, f = I.icosphere(3)
    f = f[:tris]
    cvo = wob.ControlVariate(wob.build_mesh(v, f), level=level, near=2.0)
    nodes = C.Nodes(v, f, level=level)
    fz = lambda q: q[..., 2] + 0.3 * q[..., 0] * q[..., 1] - 0.2
    v32 = [np.asarray(x, np.float32) for x in nodes.values(fz)]
    cvo.set_node_values(*v32)
    vals = [x.astype(np.float64) for x in v32]

    def bar(x, fx, own=-1):
        t = 0.0
        for pos, w, val in ((nodes.coarse_pos, nodes.coarse_w, vals[0]),
                            (nodes.fine_pos, nodes.fine_w, vals[1])):
            r = np.linalg.norm(pos - x, axis=-1)
            e = (w * (r + 2 * np.linalg.norm(pos, axis=-1)) * (np.abs(val) + abs(fx)) /
                 (4 * np.pi * r ** 3)).sum(axis=-1)
            t += e.sum() - (e[own] if own >= 0 else 0.0)
        return 32 * 2.0 ** -24 * t + 1e-7

    q = np.concatenate([I.ball_queries(points, 0.9, 3)[::2],
                        1.4 * I.ball_queries(points, 0.9, 5)[1::2] + 1.2]).astype(np.float32)
    got = cvo.quad_D(q).cpu().numpy()
    for i in range(0, len(q), max(1, len(q) // 30)):
        x = q[i].astype(np.float64)
        assert abs(got[i] - C.quad_D(nodes, vals, x, near=2.0)) <= bar(x, 0.0), (i, got[i])
    p, prim = I.boundary_points(v, f, points, 4)
    fx = fz(p.astype(np.float64)).astype(np.float32)
    got = cvo.quad_H(p, prim, fx, phi=1).cpu().numpy()
    for i in range(0, len(p), max(1, len(p) // 30)):
        x = p[i].astype(np.float64)
        want = C.quad_H(nodes, vals, x, prim[i], float(fx[i]), 1, near=2.0)
        assert abs(got[i] - want) <= 2 * bar(x, float(fx[i]), prim[i]) + 1e-6, (i, got[i], want)
