"""The line engine on trees either side of seven levels, where its node phase ends
at another share of busy lanes: the walks' values do not depend on the schedule,
so a call with a group of lanes per walk and a debug solve (a lane per walk) agree
bit for bit."""
import pytest

from paper_2305_04403_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level,depth", [(5, 5), (6, 6)])
def test_schedules_agree(level, depth):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_04403_gb300 as wob
    v, f = I.icosphere(level)
    bvh = wob.build_bvh(wob.build_mesh(v, f))
    assert bvh.info()["depth"] == depth
    prob = wob.Problem(bvh, data_mode=wob.DATA_POINT, x0=(3.0, 0.0, 0.5))
    q = I.ball_queries(37, 0.9, 3)
    est, var = wob.solve(prob, q, 65, 6, seed=5)
    dbg = wob.solve_debug(prob, q, 65, 6, seed=5, want_lines=False)
    assert torch.equal(est, dbg["est"]) and torch.equal(var, dbg["var"])
