"""(D f) off the surface with every triangle near: the near triangles' terms are
summed in FP32 over at most 64 of them, FP64 from there on.  One node value of
2^25 among ones, seen from about the centre of a sphere: the other terms t are
below half a unit of the large one's FP32 sum, so a sum that ran on in FP32
would lose all that follow it (2,560 of them in a warp's share of 20,480
triangles).  Bar: 64 lost terms, and the terms' worst-case rounding,
24 u sum w (|r| + 2 |y|) |f| / (4 pi r^3) with u = 2^-24."""
import numpy as np
import pytest

from oracle import cv as C
from paper_2305_04403_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level", [0, 1])
def test_near_sum_does_not_run_on_in_fp32(level):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_04403_gb300 as wob
    v, f = I.icosphere(5)
    cvo = wob.ControlVariate(wob.build_mesh(v, f), level=level, near=1e3)
    nodes = C.Nodes(v, f, level=level)
    vals = [np.ones(w.shape, np.float32) for w in (nodes.coarse_w, nodes.fine_w)]
    for x in vals:
        x[0] = 2.0 ** 25
    cvo.set_node_values(*vals)
    vals = [x.astype(np.float64) for x in vals]
    q = I.ball_queries(5, 0.01, 3)
    got = cvo.quad_D(q).cpu().numpy()
    for i, x in enumerate(q.astype(np.float64)):
        r = np.linalg.norm(nodes.fine_pos - x, axis=-1)
        y = np.linalg.norm(nodes.fine_pos, axis=-1)
        e = nodes.fine_w * np.abs(vals[1]) / (4 * np.pi * r ** 3)
        small = (e * r).sum(axis=-1)[1:].max()
        bar = 64 * small + 24 * 2.0 ** -24 * (e * (r + 2 * y)).sum()
        assert abs(got[i] - C.quad_D(nodes, vals, x, near=1e3)) <= bar, (i, got[i], bar)
