"""Forward paths with a group of lanes per path (calls of at most 200 paths per
SM) and with one lane per path: a path's draws depend on its index only, so the
vertices, weights and flags of the paths that a small call and a large one share
are equal bit for bit.  With a boundary that has a hole, so that lines miss and
paths end before their last record."""
import pytest

from paper_2305_04403_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("start_mode", [0, 1])
@pytest.mark.parametrize("paths,M,hole", [(2, 1, False), (33, 7, False), (1000, 5, True), (0, 4, True)])
def test_forms_agree(start_mode, paths, M, hole):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2305_04403_gb300 as wob
    edge = 200 * torch.cuda.get_device_properties(0).multi_processor_count
    v, f, _ = I.star_mesh(3, 0.3, 6, 3, 0.5)
    if hole:
        f = f[: len(f) * 2 // 3]
    prob = wob.Problem(wob.build_bvh(wob.build_mesh(v, f)), kind=wob.NEUMANN_SL, side=1,
                       data_mode=wob.DATA_POINT, x0=(3.0, 0.5, -1.0))
    q = I.ball_queries(8, 0.3, 2)
    n = paths or edge  # the largest call with groups
    a = wob.solve_forward(prob, q, n, M, seed=3, start_mode=start_mode, want_paths=True)
    b = wob.solve_forward(prob, q, edge + 33, M, seed=3, start_mode=start_mode, want_paths=True)
    for k in ("zpos", "zw", "flag"):
        assert torch.equal(a[k], b[k][:n]), k
    ended = int((a["zw"][:, -1] == 0).sum())
    assert (ended > 0) == hole or n < 1000, ended
