"""The limits at which the GPU triangulation answers "failed" (*ntri = -1) in
place of a mesh: no room in the pool for the triangles of large fans, and
points too far apart for its integer steps; just inside both, the mesh."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import dev, host, require_gpu, torch

pytestmark = pytest.mark.gpu

SLOTS = 16  # owned triangles that a point keeps outside the pool


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _canon(t):
    return sorted(tuple(int(v) for v in np.roll(r, -int(np.argmin(r)))) for r in np.asarray(t).reshape(-1, 3))


def _run(lst, w, h, right=False, pool=None):
    """The mesh (None: failed) and the workspace, which held 0xA5 before the call."""
    from paper_1802_07210_gb300 import binding as B
    L = B.lib()
    cap = len(lst)
    d, cnt = dev(np.asarray(lst, np.int16)), dev(np.array([cap], np.int32))
    tri = torch.empty((2 * cap + 8, 3), dtype=torch.int32, device="cuda")
    nt = torch.zeros(1, dtype=torch.int32, device="cuda")
    nb = L.elas_triangulate_device_workspace_bytes(cap, w, h)
    ws = torch.full((nb,), 0xA5, dtype=torch.uint8, device="cuda")
    args = [d.data_ptr(), cnt.data_ptr(), cap, w, h, int(right), tri.data_ptr(), 2 * cap + 8, nt.data_ptr(),
            ws.data_ptr(), nb]
    st = torch.cuda.current_stream().cuda_stream
    B.check(L.elas_triangulate_device(*args, st) if pool is None else
            L.elas_probe_triangulate_pool(*args, pool, st))
    k = int(host(nt)[0])
    assert k >= -1
    return (None if k < 0 else host(tri)[:k]), host(ws)


def _pool_bytes(ws, cap, h):
    """The pool's 2 cap entries: in the workspace they lie before the two queues, the row extremes
    and the counters."""
    def up(b):
        return (b + 255) // 256 * 256
    end = len(ws) - up(20) - 2 * up(4 * h) - 2 * up(4 * cap)
    return ws[end - up(16 * cap):][:16 * cap]


@pytest.mark.parametrize("fan", [26, 255, 700])
def test_pool_without_room(fan):
    """An apex that sees every point of a distant row, certain to a warp (26), wrapped by a CTA over its
    cached points and by a CTA over all points (more vertices than its lists hold)."""
    if fan == 26:  # the points of a half ring within a warp's 24 pixels that the apex sees
        ring = [(x, y) for y in range(1, 25) for x in range(-24, 25) if 22 * 22 <= x * x + y * y <= 24 * 24]
        lst = np.array([(100, 40, 3)] + [(100 + x, 40 + y, 3) for x, y in ring], np.int16)
        t = oracle.triangulate(lst)
        lst, w, h = lst[np.unique(t[(t == 0).any(1)])], 200, 100
    else:
        lst = [(2, 3, 1)] + [(10 + 5 * i, 900, 1 + i % 7) for i in range(fan)]
        w, h = 5 * fan + 20, 910
    lst = np.array(lst, np.int16)
    exp = oracle.triangulate(lst)
    owned = np.bincount(exp.min(1), minlength=len(lst))
    need = int(owned[owned > SLOTS].sum())
    assert need > 0
    for pool in (2 * len(lst), need):
        got, ws = _run(lst, w, h, pool=pool)
        assert got is not None and _canon(got) == _canon(exp)
        used = _pool_bytes(ws, len(lst), h)
        assert (used[8 * need:] == 0xA5).all() and (used[:8 * need].view(np.int32) < len(lst)).all()
    for pool in (need - 1, SLOTS, 0):
        got, ws = _run(lst, w, h, pool=pool)
        assert got is None
        assert (_pool_bytes(ws, len(lst), h)[8 * pool:] == 0xA5).all()


def _spread(n, x0, x1, h, seed):
    """n points over the x extent [x0, x1] of right coordinates (u - d) and all of [0, h)."""
    rng = np.random.default_rng(seed)
    x = np.concatenate([[x0, x1, x0, x1], rng.integers(x0, x1 + 1, n - 4)])
    v = np.concatenate([[0, 0, h - 1, h - 1], rng.integers(0, h, n - 4)])
    at = np.lexsort((x, v))
    x, v = x[at], v[at]
    u = np.clip(x, -32768, 32767)
    d = u - x
    assert (np.abs(d) <= 32767).all()
    return np.stack([u, v, d], 1).astype(np.int16)


# h = 16,001: Y = 16,000, so X up to sqrt(2^31 - 1 - Y^2) = 43,491
@pytest.mark.parametrize("x0,x1,ok", [
    (0, 16382, True),          # an image
    (-1023, 16382, True),      # and its disparities
    (-8192, 32767, True),      # the corners of the box that needs no look at the extents
    (-8193, 32767, True),      # outside it
    (-32768, -20000, True),    # all of it
    (-10724, 32767, True),     # X = 43,491
    (-10725, 32767, False),
    (-32768, 32767, False),
    (-60000, 60000, False),
])
@pytest.mark.parametrize("n", [40, 400])
def test_extents(x0, x1, ok, n):
    lst = _spread(n, x0, x1, 16001, n)
    got, _ = _run(lst, 16383, 16001, right=True)
    if ok:
        assert got is not None and _canon(got) == _canon(oracle.triangulate(lst, right=True))
    else:
        assert got is None


def test_extents_in_a_batch_of_sides():
    """One pair's list whose left points fit and whose right ones do not: each call by itself."""
    lst = _spread(60, -30000, 32767, 500, 3)
    left, _ = _run(lst, 16383, 500, right=False)
    right, _ = _run(lst, 16383, 500, right=True)
    assert left is None and right is None  # u alone spans 62,767
    lst[:, 0] = np.clip(lst[:, 0], 0, 32767)
    lst = np.unique(lst, axis=0)
    lst = lst[np.lexsort((lst[:, 0], lst[:, 1]))]
    got, _ = _run(lst, 16383, 500, right=False)
    assert got is not None and len(got) > 0
