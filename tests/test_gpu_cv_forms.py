"""(D f) off the surface in every form of its kernel, against the FP64 quadrature:
triangles near to few and to most points of a warp (summed for queued pairs, or by
every lane for its own point), eight warps to 32 points and a set per warp (calls
of many points).  A point's value does not depend on which points are beside it.

Bar: the terms' worst-case rounding, 24 u sum w (|r| + 2 |y|) |f| / (4 pi r^3) with
u = 2^-24, and 8 u of it for the FP32 sums."""
import numpy as np
import pytest

from oracle import cv as C
from paper_2305_04403_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh,tris,level,near,points", [
    (0, 20, 0, 8.0, 33), (0, 20, 0, 2.0, 100000), (0, 19, 1, 2.0, 300001), (1, 80, 1, 2.0, 300000),
    (1, 80, 2, 8.0, 300), (2, 320, 3, 8.0, 65), (3, 1279, 2, 1.0, 3000), (3, 1280, 0, 4.0, 300033)])
def test_forms(mesh, tris, level, near, points):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_04403_gb300 as wob
    v, f = I.icosphere(mesh)
    f = f[:tris]
    cvo = wob.ControlVariate(wob.build_mesh(v, f), level=level, near=near)
    nodes = C.Nodes(v, f, level=level)
    fz = lambda q: q[..., 2] + 0.3 * q[..., 0] * q[..., 1] - 0.2
    v32 = [np.asarray(x, np.float32) for x in nodes.values(fz)]
    cvo.set_node_values(*v32)
    vals = [x.astype(np.float64) for x in v32]
    q = I.ball_queries(points, 0.7, 3).astype(np.float32)
    q[1::2] += np.float32(1.3)
    got = cvo.quad_D(q).cpu().numpy()
    pick = np.unique(np.linspace(0, points - 1, 24).astype(int))
    alone = cvo.quad_D(q[pick]).cpu().numpy()
    for k, i in enumerate(pick):
        x = q[i].astype(np.float64)
        t = 0.0
        for pos, w, val in ((nodes.coarse_pos, nodes.coarse_w, vals[0]),
                            (nodes.fine_pos, nodes.fine_w, vals[1])):
            r = np.linalg.norm(pos - x, axis=-1)
            t += (w * (r + 2 * np.linalg.norm(pos, axis=-1)) * np.abs(val) / (4 * np.pi * r ** 3)).sum()
        bar = 32 * 2.0 ** -24 * t + 1e-7
        want = C.quad_D(nodes, vals, x, near=near)
        assert abs(got[i] - want) <= bar and abs(alone[k] - want) <= bar, (i, got[i], alone[k], want)
