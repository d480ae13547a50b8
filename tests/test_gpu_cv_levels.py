"""Control variates of several subdivision levels side by side: what one
computes does not depend on which others exist.  The quadrature H, the nodes
and the residual walks of an object that was alone, and again after objects of
the other levels were created, are equal bit for bit."""
import numpy as np
import pytest

from paper_2305_04403_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level", [0, 1, 2, 3])
def test_levels_side_by_side(level):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_04403_gb300 as wob
    v, f = I.icosphere(2)
    mesh = wob.build_mesh(v, f)
    prob = wob.Problem(wob.build_bvh(mesh), data_mode=wob.DATA_POINT, x0=(0.0, 0.0, 3.0))
    params = wob.mlp_init(3)
    p, prim = I.boundary_points(v, f, 200, 4)
    q = I.ball_queries(16, 0.8, 3)

    def results(cvo):
        s, s2 = (torch.zeros(len(q), dtype=torch.float64, device="cuda") for _ in range(2))
        cvo.solve_range(prob, params, q, 0, 16, 3, s, s2, seed=1)
        return [cvo.quad_H(p, prim, np.ones(len(p), np.float32), phi=1), *cvo.nodes(), s, s2]

    cvo = wob.ControlVariate(mesh, level=level, near=2.0)
    cvo.set_network(params)
    alone = results(cvo)
    others = [wob.ControlVariate(mesh, level=n, near=2.0) for n in range(4) if n != level]
    for got, want in zip(results(cvo), alone):
        assert torch.equal(torch.as_tensor(got), torch.as_tensor(want))
    assert len(others) == 3
