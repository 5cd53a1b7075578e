"""The kernels that a size, a type or an alignment picks, at the edges of
their tiles and of the rules, against the oracle: support matching by parts of
lattice rows, the 3x3 median and small-segment removal (word accesses or not),
the LR check (one or two pixels an access), the fused post-processing tile and
the prior of triangles much larger than the units they are drawn in, and chains
of calls whose kernels start early."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import dev, grid_as_i32, host, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _B():
    from paper_1802_07210_gb300 import binding
    return binding


def _at(a, offset):
    """a on the GPU, `offset` elements past an aligned address."""
    t = torch.empty(a.size + offset, dtype=torch.from_numpy(a[:1]).dtype, device="cuda")
    v = t[offset:].view(a.shape)
    v.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return v


def _map(w, h, holes, top=60, seed=0):
    rng = np.random.default_rng(1000 * w + h + seed)
    d = (np.add.outer(np.arange(h) // 9, np.arange(w) // 13) * 3 + rng.integers(-1, 2, (h, w))) % top
    d = d.astype(np.int16)
    d[rng.random((h, w)) < holes] = -1
    return d


# sizes around the 64x16 and (from 152 tiles on) 64x32 tiles, even and odd widths
FILTER_SIZES = [(1, 1), (2, 1), (63, 15), (64, 16), (65, 17), (66, 31), (128, 32), (129, 33), (190, 65), (1217, 257)]


@pytest.mark.parametrize("size", FILTER_SIZES)
@pytest.mark.parametrize("offset", [0, 1, 2])
def test_median_3x3(size, offset):
    """No holes, some, mostly holes; values of the whole range of disparities."""
    B = _B()
    w, h = size
    for holes in (0.0, 0.1, 0.7):
        d = _map(w, h, holes)
        wide = np.random.default_rng(w + h).integers(0, 1024, (h, w)).astype(np.int16)
        wide[d < 0] = -1
        for m in (d, wide):
            out = _at(np.zeros_like(m), offset)
            B.elas_median(_at(m, offset), 1, out=out)
            np.testing.assert_array_equal(host(out), oracle.median(m, 1))


@pytest.mark.parametrize("size", FILTER_SIZES)
@pytest.mark.parametrize("offset", [0, 1, 4])
def test_speckle_tiles(size, offset):
    B = _B()
    w, h = size
    for holes, thr, least in ((0.0, 1, 40), (0.2, 1, 12), (0.45, 2, 5), (0.1, 0, 3)):
        d = _map(w, h, holes, seed=thr)
        out = _at(np.zeros_like(d), offset)
        _, st = B.elas_speckle(_at(d, offset), thr, least, out=out, with_status=True)
        np.testing.assert_array_equal(host(out), oracle.speckle(d, thr, least))
        assert int(host(st)[0]) == 0


@pytest.mark.parametrize("w", [1, 2, 31, 255, 256, 770, 1537, 1538])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("masks", [False, True])
def test_lr_check_widths(w, offset, masks):
    B = _B()
    l, r = _map(w, 5, 0.1), _map(w, 5, 0.1, seed=1)
    for thr in (0, 2):
        dL, dR = _at(l, offset), _at(r, offset)
        got = B.elas_lr_check(dL, dR, thr, masks=masks)
        el, er, ml, mr = oracle.lr_check(l, r, thr)
        np.testing.assert_array_equal(host(dL), el)
        np.testing.assert_array_equal(host(dR), er)
        if masks:
            np.testing.assert_array_equal(host(got[0]), ml)
            np.testing.assert_array_equal(host(got[1]), mr)


@pytest.mark.parametrize("size", [(1, 1), (31, 23), (32, 24), (33, 25), (65, 49), (97, 71)])
@pytest.mark.parametrize("gap,mean", [(0, 1), (1, 1), (2, 1), (3, 1), (3, 0), (4, 1), (16, 1)])
def test_fused_post_tiles(size, gap, mean):
    """A weight of the mean is a small multiple of 1/4 and a sum of 8 products
    below 2^10: each FP32 operation is off by at most 2^-24 of it, some 20 of
    them in a pass over values up to 60 by less than 1e-4."""
    w, h = size
    prm = dict(ipol_gap_width=gap, filter_adaptive_mean=mean)
    d = _map(w, h, 0.25)
    exp = oracle.postprocess(d, prm)
    out = host(_B().elas_postprocess(dev(d), prm))
    assert np.abs(out - exp).max() <= 1e-4
    assert ((out < 0) == (exp < 0)).all()


def _support(w, h, prm):
    rng = np.random.default_rng(w * h)
    # texture shifted by a disparity that grows down the image, some noise
    base = rng.integers(0, 256, (h, w + 64)).astype(np.int32)
    base = (base + np.roll(base, 1, 1) + np.roll(base, 1, 0)) // 3
    shift = 5 + (np.arange(h) * 20) // max(h, 1)
    L = base[:, :w]
    R = np.stack([base[y, s:s + w] for y, s in enumerate(shift)]) + rng.integers(-2, 3, (h, w))
    return L.astype(np.uint8), np.clip(R, 0, 255).astype(np.uint8)


# lattices on both sides of each limit: 32,768 candidates; 304 lattice rows;
# rows of fewer than 16 candidates, of a whole number of parts and ragged ones
@pytest.mark.parametrize("w,h,step,d", [
    (410, 320, 2, 64),    # 32,800 candidates: eight parts of a row
    (406, 320, 2, 64),    # 32,480: a warp per candidate
    (401, 333, 2, 130),   # ragged parts, two words of disparity bits and more
    (257, 140, 1, 40),    # step 1, an odd lattice width
    (40, 310, 1, 20),     # 310 rows, two parts each
    (14, 320, 1, 6),      # rows too short for a part
    (720, 460, 3, 200),   # parts narrower than the disparity range
])
@pytest.mark.parametrize("census", [False, True])
def test_support_by_row_parts(w, h, step, d, census):
    B = _B()
    prm = dict(disp_max=d - 1, candidate_stepsize=step)
    if census:
        prm.update(census_support_w=9, census_dense_w=5, beta=0.1)
    L, R = _support(w, h, prm)
    if census:
        descL, descR = oracle.census(L, 9, 32), oracle.census(R, 9, 32)
    else:
        descL, descR = oracle.descriptors(L), oracle.descriptors(R)
    exp = oracle.support_points(descL, descR, prm)
    lst = oracle.support_list(exp, prm)
    r = B.elas_support_points(dev(descL), dev(descR), prm)
    np.testing.assert_array_equal(host(r["d_can"]), exp)
    n = int(host(r["count"])[0])
    assert n == len(lst) and n > 0
    np.testing.assert_array_equal(host(r["list"])[:n], lst)
    np.testing.assert_array_equal(host(r["grid_L"]), grid_as_i32(oracle.grid_vectors(lst, w, h, prm)))
    np.testing.assert_array_equal(host(r["grid_R"]), grid_as_i32(oracle.grid_vectors(lst, w, h, prm, right=True)))


@pytest.mark.parametrize("maxd", [1, 5, 60])
@pytest.mark.parametrize("size", [(205, 120), (210, 120), (240, 120)])
def test_redundancy_rows(size, maxd):
    """Row staging by 2, 4 and 16 bytes (41, 42 and 48 candidates a row), few
    and many rows of it, disparities that cross the words of the bit vectors."""
    w, h = size
    prm = dict(disp_max=99, redun_max_dist=maxd, grid_size=7)
    L, R = _support(w, h, prm)
    descL, descR = oracle.descriptors(L), oracle.descriptors(R)
    exp = oracle.support_points(descL, descR, prm)
    lst = oracle.support_list(exp, prm)
    r = _B().elas_support_points(dev(descL), dev(descR), prm)
    np.testing.assert_array_equal(host(r["d_can"]), exp)
    np.testing.assert_array_equal(host(r["grid_L"]), grid_as_i32(oracle.grid_vectors(lst, w, h, prm)))
    np.testing.assert_array_equal(host(r["grid_R"]), grid_as_i32(oracle.grid_vectors(lst, w, h, prm, right=True)))


@pytest.mark.parametrize("n", [3, 4, 9, 60])
@pytest.mark.parametrize("right", [False, True])
def test_prior_of_few_large_triangles(n, right):
    """Triangles across the whole map, slivers along its edges among them."""
    w, h = 701, 403
    rng = np.random.default_rng(n)
    pts = np.unique(np.stack([rng.integers(70, w, n), rng.integers(0, h, n)], 1), axis=0)
    pts = np.concatenate([pts, [[70, 0], [w - 1, 1], [w - 1, h - 1]]])
    pts = np.unique(pts, axis=0)
    pts = pts[np.lexsort((pts[:, 0], pts[:, 1]))]
    lst = np.concatenate([pts, rng.integers(0, 64, (len(pts), 1))], 1).astype(np.int16)
    prm = dict(disp_max=63)
    tri = oracle.triangulate(lst, right=right).astype(np.int32)
    exp = oracle.plane_prior(lst, tri, w, h, prm, right=right)
    out = _B().elas_plane_prior(dev(lst), dev(tri), w, h, prm, right=right)
    np.testing.assert_array_equal(host(out), exp)


def _calls(B, L, R, prm, stream=None):
    """Every single-stage call of a pair after the other, as a program without
    the pipeline makes them (capacities in place of counts: no copy to the host)."""
    dl, dr = B.elas_descriptors(L, R, stream=stream)
    s = B.elas_support_points(dl, dr, prm, stream=stream)
    h, w = L.shape
    tri = [B.elas_triangulate_device(s["list"], s["count"], w, h, right, stream=stream) for right in (False, True)]
    d = B.elas_dense_argmin(dl, dr, dict(prm, flags=2), stream=stream)
    dR = B.elas_dense_argmin(dl, dr, dict(prm, flags=2), right=True, stream=stream)
    B.elas_lr_check(d, dR, 2, masks=False, stream=stream)
    post = B.elas_postprocess(d, prm, stream=stream)
    return [s["d_can"], s["count"], s["grid_L"], s["grid_R"], tri[0][1], tri[1][1], d, dR, post,
            B.elas_median(d, 1, stream=stream), B.elas_speckle(d, 1, 20, stream=stream)]


def test_chains_of_calls_on_streams_and_captured():
    """The calls' kernels may take their places before the one ahead of them
    ends: chains over changing inputs, queued without a stop on one stream, on
    two streams in turn and replayed from a graph, give what a chain with a
    synchronisation after it gives."""
    B = _B()
    prm = dict(disp_max=47, ipol_gap_width=3, filter_adaptive_mean=1)
    pairs = [tuple(dev(a) for a in _support(203 + 64 * k, 117, prm)) for k in range(3)]
    alone = []
    for L, R in pairs:
        alone.append([t.clone() for t in _calls(B, L, R, prm)])
        torch.cuda.synchronize()
    got = [(k % 3, _calls(B, *pairs[k % 3], prm)) for k in range(24)]
    side = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    for k in range(24):
        with torch.cuda.stream(side[k % 2]):
            got.append((k % 3, _calls(B, *pairs[k % 3], prm)))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side[0]):
        out = _calls(B, *pairs[1], prm, stream=side[0])
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    got.append((1, out))
    for k, res in got:
        for a, b in zip(res, alone[k]):
            np.testing.assert_array_equal(host(a), host(b))


@pytest.mark.parametrize("size", [(65, 49), (97, 71), (200, 30)])
@pytest.mark.parametrize("gap", [6, 7, 8, 9, 10, 11, 13, 15, 16])
@pytest.mark.parametrize("mean", [0, 1])
def test_wide_gaps(size, gap, mean):
    """Holes of every length around the gap width, along rows and columns, the search in steps
    (up to 7) and in fours (from 8 on).  The tolerance is test_fused_post_tiles's."""
    w, h = size
    prm = dict(ipol_gap_width=gap, filter_adaptive_mean=mean)
    rng = np.random.default_rng(gap)
    d = _map(w, h, 0.05)
    for k in range(60):
        x, y, n = rng.integers(0, w), rng.integers(0, h), rng.integers(max(1, gap - 3), gap + 3)
        if k % 2:
            d[y, x:x + n] = -1
        else:
            d[y:y + n, x:x + 3] = -1
    exp = oracle.postprocess(d, prm)
    out = host(_B().elas_postprocess(dev(d), prm))
    assert np.abs(out - exp).max() <= (1e-4 if mean else 0)
    assert ((out < 0) == (exp < 0)).all()


@pytest.mark.parametrize("size", [(20, 1500), (100, 700), (700, 100), (641, 479)])
@pytest.mark.parametrize("shape", ["comb", "comb_top", "comb_right", "snake", "rings"])
def test_speckle_long_segments(size, shape):
    """Segments that run through many tiles and meet at one end, so that the links across the
    tiles' edges form long chains."""
    B = _B()
    w, h = size
    d = np.full((h, w), -1, np.int16)
    if shape == "comb":
        d[:, ::2], d[-1] = 5, 5
    elif shape == "comb_top":
        d[:, ::2], d[0] = 5, 5
    elif shape == "comb_right":
        d[::2], d[:, -1] = 5, 5
    elif shape == "snake":
        d[::2], d[1::4, -1], d[3::4, 0] = 5, 5, 5
    else:
        y, x = np.mgrid[:h, :w]
        d[np.minimum(np.minimum(x, w - 1 - x), np.minimum(y, h - 1 - y)) % 2 == 0] = 5
    for least in (10, w * h // 3):
        for _ in range(3):
            out, st = B.elas_speckle(dev(d), 1, least, with_status=True)
            np.testing.assert_array_equal(host(out), oracle.speckle(d, 1, least))
            assert int(host(st)[0]) == 0


@pytest.mark.parametrize("size", [(1, 1), (31, 23), (33, 25), (640, 41)])
@pytest.mark.parametrize("offset", [0, 1])
def test_post_without_passes(size, offset):
    """Neither gap interpolation nor means: the map's own values as floats."""
    B = _B()
    w, h = size
    d = _map(w, h, 0.2)
    d[d < 0] = np.random.default_rng(3).choice([-1, -2, -300], (d < 0).sum())
    out = host(B.elas_postprocess(_at(d, offset), dict(ipol_gap_width=0, filter_adaptive_mean=0)))
    np.testing.assert_array_equal(out, d.astype(np.float32))
