"""The tree's sort either side of its shared-memory chunk (4,096 triangles, and
past two of them), by the triangles that lines hit, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2305_04403_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wob():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_04403_gb300 as w
    return w


@pytest.mark.parametrize("tris", [1, 2, 3, 4095, 4096, 4097, 8193, 16385, 20480])
def test_sorted_tree_hits(wob, tris):
    v, f = I.icosphere(5)
    f = f[:tris]
    q = I.ball_queries(64, 0.9, 3)
    prob = wob.Problem(wob.build_bvh(wob.build_mesh(v, f)), kind=wob.DIRICHLET_DL, side=1,
                       data_mode=wob.DATA_POLY, poly=I.POLY_CONFIG1)
    g = wob.solve_debug(prob, q, 32, 2, seed=4)
    r = O.dl_walks(v, f, q, 32, 2, seed=4, poly=I.POLY_CONFIG1, want_lines=True)
    ok = (g["flag"].cpu().numpy() == 0) & (r["flag"] == 0)
    assert ok.mean() > 0.95
    assert np.array_equal(g["line_m"].cpu().numpy()[ok], r["line_m"][ok])
    assert np.array_equal(g["line_prim"].cpu().numpy()[ok], r["line_prim"][ok])
