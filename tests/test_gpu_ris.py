"""Resampled single-layer walks on boundaries of very small and very large extent
and on candidates that are nearly all close to the vertex, against the oracle."""
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


@pytest.mark.parametrize("kind,alpha", [(1, 0.0), (2, 0.5)])
@pytest.mark.parametrize("size", [1e-6, 1.0, 1e6])
def test_ris_extent(wob, kind, alpha, size):
    """Bar: 1e-5 of the sum of |term|, as at unit size."""
    v, f = I.icosphere(2)
    v = (v * size).astype(np.float32)
    q = (I.ball_queries(16, 0.8, 3) * size).astype(np.float32)
    x0 = (0.0, 0.0, 3.0 * size)
    prob = wob.Problem(wob.build_bvh(wob.build_mesh(v, f)), kind=kind, side=1, alpha=alpha / size,
                       data_mode=wob.DATA_POINT, x0=x0, ris=8)
    g = wob.solve_debug(prob, q, 64, 4, seed=2, want_lines=False)["per_walk"].cpu().numpy()
    pw, at = O.sl_walks(v, f, q, 64, 4, kind=kind, alpha=alpha / size, phi=1, mode=O.DATA_POINT,
                        x0=x0, seed=2, want_abs=True, ris=8)
    assert np.all(np.abs(g - pw) <= 1e-5 * at)


def test_ris_close_candidates(wob):
    """Queries 1e-3 to 1e-6 off the surface of one large triangle's fan: the
    query's candidates of that triangle are close ones, up to 64 of them."""
    v, f = I.icosphere(0)
    p, _ = I.boundary_points(v, f, 32, 4)
    q = (p * (1 - 10.0 ** -np.linspace(3, 6, 32))[:, None]).astype(np.float32)
    x0 = (0.0, 0.0, 3.0)
    prob = wob.Problem(wob.build_bvh(wob.build_mesh(v, f)), kind=1, side=1,
                       data_mode=wob.DATA_POINT, x0=x0, ris=64)
    g = wob.solve_debug(prob, q, 256, 2, seed=2, want_lines=False)["per_walk"].cpu().numpy()
    pw, at = O.sl_walks(v, f, q, 256, 2, kind=1, phi=1, mode=O.DATA_POINT, x0=x0, seed=2,
                        want_abs=True, ris=64)
    assert np.all(np.abs(g - pw) <= 1e-5 * at)
