"""The two forms of the line engine (one lane per walk, and a group of lanes
per walk for calls with few walks) against each other and the oracle: debug
solves always take the first, plain solves of few walks the second.  The
values of the walks are the same numbers and are summed in the same order,
so the estimates are equal bit for bit."""
import os
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))

import oracle as O  # noqa: E402
import paper_2305_04403_gb300 as wob  # noqa: E402
from _parity import compare_walks  # noqa: E402
from paper_2305_04403_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


def _shells(n):
    """n nested spheres (a line near the centre meets all of them twice)."""
    v, f = I.icosphere(2)
    r = 0.4 + 0.6 * np.arange(n) / n
    return (np.concatenate([v * x for x in r]).astype(np.float32),
            np.concatenate([f + i * len(v) for i in range(n)]).astype(np.int32))


# tile remainders, a single query, the largest grouped call and one beyond it
# (a call of at most 200 walks per SM runs with a group of lanes per walk)
@pytest.mark.parametrize("Q,N,M", [(1, 2, 1), (3, 33, 5), (17, 31, 3), (1, 65, 24), (0, 64, 3),
                                   (-1, 64, 3)])
@pytest.mark.parametrize("mesh", ["torus", "shells"])
@pytest.mark.parametrize("kind", [wob.DIRICHLET_DL, wob.NEUMANN_DIRECT])
def test_forms_agree(Q, N, M, mesh, kind):
    if Q < 1:  # around the line between the two forms
        Q = 200 * torch.cuda.get_device_properties(0).multi_processor_count // N - Q
    v, f = I.displaced_torus(30, 12)[:2] if mesh == "torus" else _shells(6)
    q, prim = I.boundary_points(v, f, Q, 3)
    q = (0.97 * q).astype(np.float32)
    bvh = wob.build_bvh(wob.build_mesh(v, f), leaf_size=1 if N % 2 else 3)
    prob = wob.Problem(bvh, kind=kind, data_mode=wob.DATA_POINT, x0=(3.0, 0.0, 0.5))
    est, var = wob.solve(prob, q, N, M, seed=5)
    dbg = wob.solve_debug(prob, q, N, M, seed=5, want_lines=False)
    assert torch.equal(est, dbg["est"]) and torch.equal(var, dbg["var"])
    if kind == wob.DIRICHLET_DL:  # gradients: the same queries alone and first among many
        n = 201 * torch.cuda.get_device_properties(0).multi_processor_count // N
        many = np.concatenate([q, np.repeat(q[:1], max(0, n + 1 - Q), 0)])
        a, b = (wob.solve_grad(prob, x, N, M, seed=5) for x in (q, many))
        assert all(torch.equal(a[k], b[k][..., :Q]) for k in a)


def test_more_hits_than_recorded():
    """Twelve crossings a line: the pick keeps a running minimum of the keys
    beyond the recorded hits; every line against the oracle's."""
    v, f = _shells(6)
    q = I.ball_queries(24, 0.3, 7)
    prob = wob.Problem(wob.build_bvh(wob.build_mesh(v, f)), data_mode=wob.DATA_POINT,
                       x0=(3.0, 0.0, 0.5))
    g = {k: t.cpu().numpy() for k, t in wob.solve_debug(prob, q, 33, 3, seed=2).items()}
    r = O.dl_walks(v, f, q, 33, 3, seed=2, mode=O.DATA_POINT, x0=(3.0, 0.0, 0.5), want_lines=True)
    assert g["line_m"].max() == 12
    same, _ = compare_walks(g, r, 1.0)
    assert same.mean() > 0.98
    est, _ = wob.solve(prob, q, 33, 3, seed=2)
    assert np.array_equal(est.cpu().numpy(), g["est"])
