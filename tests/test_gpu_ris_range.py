"""Resampled single-layer walks at the ends of FP32's range, against the FP64
oracle: exterior queries far from the boundary (r^2 in units of its extent leaves
the range, 1 / r loses its low part before), very small and large boundaries and a
very large Robin coefficient.  Bar: 1e-5 of the sum of |term|, as at ordinary
sizes."""
import numpy as np
import pytest

import oracle as O
from paper_2305_04403_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(kind, alpha, side, size, q):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_04403_gb300 as wob
    v, f = I.icosphere(2)
    vd = (1.0 + 0.5 * v[:, 2] + 0.25 * v[:, 0] * v[:, 1]).astype(np.float32)
    v = (v * np.float64(size)).astype(np.float32)
    prob = wob.Problem(wob.build_bvh(wob.build_mesh(v, f)), kind=kind, side=side, alpha=alpha,
                       data_mode=wob.DATA_VERTEX_P1, vertex_data=vd, ris=8)
    g = wob.solve_debug(prob, q, 64, 3, seed=2, want_lines=False)["per_walk"].cpu().numpy()
    pw, at = O.sl_walks(v, f, q, 64, 3, kind=kind, alpha=alpha, phi=side, mode=O.DATA_VERTEX_P1,
                        vertex_data=vd, seed=2, want_abs=True, ris=8)
    assert np.isfinite(pw).all() and (at > 0).all()
    assert np.all(np.abs(g - pw) <= 1e-5 * at), (np.abs(g - pw) / at).max()


@pytest.mark.parametrize("kind,alpha", [(1, 0.0), (2, 0.5)])
@pytest.mark.parametrize("size,dist", [(1.0, 1e8), (1.0, 1e10), (1.0, 1e20), (1.0, 1e38), (1e-6, 1e18),
                                       (1e6, 1e37)])
def test_far_queries(kind, alpha, size, dist):
    q = I.ball_queries(16, 0.8, 3).astype(np.float64)
    q = (q / np.linalg.norm(q, axis=1, keepdims=True) * dist).astype(np.float32)
    _check(kind, alpha / size, -1, size, q)


@pytest.mark.parametrize("kind,alpha,size", [(1, 0.0, 1e-24), (1, 0.0, 1e24), (2, 0.5, 1e-24),
                                             (2, 0.5, 1e24), (2, 1e25, 1.0)])
def test_extreme_sizes(kind, alpha, size):
    q = (I.ball_queries(16, 0.8, 3) * np.float64(size)).astype(np.float32)
    _check(kind, alpha / size, 1, size, q)
