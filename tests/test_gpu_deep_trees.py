"""Trees of more than 48 levels (at most 63 can be built), whose traversal stacks
take most of the 48 KB a kernel may use: solves of two such boundaries from two
threads at once, each with its own stream, give what either gives alone."""
import ctypes
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2305_04403_gb300 as wob  # noqa: E402
from paper_2305_04403_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


def _deep(groups):
    """`groups` + 1 sets of seven equal triangles about a point whose Morton code
    alternates: set d differs from it in the code's bit d, and is larger than
    all later ones together, so a wide node holds one set and the rest."""
    top, code = 21, sum(1 << b for b in range(0, 21, 2))
    tri = [[[0, 0, 1], [1, 1, 0], [1, 0, 0]]]  # spans the unit cube
    pattern = np.array([[0, 0, 1], [0, 1, 0], [1, 0, 0]]) - 1.0 / 3.0
    for d in range(1, groups + 1):
        p = [code] * 3
        if d < groups:
            p[d % 3] ^= 1 << (top - 1 - d // 3)
        c = (np.array(p) + 0.5) / ((1 << top) - 1)
        size = min(0.999 * min(3 * c.min(), 1.5 * (1 - c).min()), 0.05 + 4.0 * 2.0 ** (-d / 3))
        tri.append(c + size * pattern)
    v = np.repeat(np.array(tri, float), 7, 0).reshape(-1, 3).astype(np.float32)
    f = np.arange(len(v), dtype=np.int32).reshape(-1, 3)
    a, b, c = (v[f[:, i]].astype(float) for i in range(3))
    return v, f if np.einsum("ij,ij->i", a, np.cross(b, c)).sum() > 0 else f[:, ::-1].copy()


@pytest.fixture(scope="module")
def problems():
    out = []
    for groups in (56, 60):
        v, f = _deep(groups)
        bvh = wob.build_bvh(wob.build_mesh(v, f))
        assert bvh.info()["depth"] >= 48
        out.append(wob.Problem(bvh, data_mode=wob.DATA_POINT, x0=(3.0, 0.0, 0.5)))
    return out


def test_two_threads(problems):
    n = 201 * torch.cuda.get_device_properties(0).multi_processor_count // 32 + 1
    q = torch.as_tensor(0.4 + 0.2 * I.ball_queries(n, 0.9, 3), dtype=torch.float32, device="cuda")
    want = [wob.solve(p, q, 32, 1, seed=2) for p in problems]
    torch.cuda.synchronize()
    failed = []
    lib = wob.load_library()

    def work(i):
        try:
            s = torch.cuda.Stream()
            got = [torch.empty_like(x) for x in want[i]]
            call = (ctypes.byref(problems[i]._c()), ctypes.c_void_p(q.data_ptr()), None, n, 32, 1, 2,
                    ctypes.c_void_p(got[0].data_ptr()), ctypes.c_void_p(got[1].data_ptr()),
                    ctypes.c_void_p(s.cuda_stream))
            for _ in range(4000):  # the C entry point: little time outside it
                rc = lib.wob_solve(*call)
                assert rc == 0, lib.wob_last_error()
            s.synchronize()
            assert torch.equal(got[0], want[i][0]) and torch.equal(got[1], want[i][1])
        except Exception as e:  # noqa: BLE001
            failed.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i % 2,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
