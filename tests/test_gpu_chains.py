"""Chains of single-stage calls whose kernels may take their places before the
one ahead of them ends, compared whole (support list, both meshes, prior and
dense match over the meshes, filters) with the same chain run with a stop after
every call, for a Sobel and a census pair: queued on one stream, on two streams
in turn and replayed from a graph."""
import numpy as np
import pytest

from tests.gpu_util import dev, host, require_gpu, torch

pytestmark = pytest.mark.gpu

PRM = dict(disp_max=47, ipol_gap_width=3, filter_adaptive_mean=1)
CENSUS = dict(PRM, census_support_w=9, census_dense_w=5, beta=0.1)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _pair(w, h, seed):
    rng = np.random.default_rng(seed)
    base = rng.integers(0, 256, (h, w + 64)).astype(np.int32)
    base = (base + np.roll(base, 1, 1) + np.roll(base, 1, 0)) // 3
    shift = 5 + (np.arange(h) * 30) // h
    L = base[:, :w]
    R = np.stack([base[y, s:s + w] for y, s in enumerate(shift)]) + rng.integers(-2, 3, (h, w))
    return dev(L.astype(np.uint8)), dev(np.clip(R, 0, 255).astype(np.uint8))


def _chain(L, R, prm, counts=None, stop=False):
    """Every output of the chain.  counts: points and triangles of the meshes, known from a run
    before (None: read from the device, which needs the stop).  The inputs of a call are what the
    call before it wrote, so a kernel that starts before they are there reads something else."""
    from paper_1802_07210_gb300 import binding as B

    def done(x):
        if stop:
            torch.cuda.synchronize()
        return x

    h, w = L.shape
    if prm.get("census_support_w"):
        sl, sr = done(B.elas_census(L, R, prm["census_support_w"], 32))
        dl, dr = done(B.elas_census(L, R, prm["census_dense_w"], 16))
    else:
        sl, sr = dl, dr = done(B.elas_descriptors(L, R))
    s = done(B.elas_support_points(sl, sr, prm))
    tri = [done(B.elas_triangulate_device(s["list"], s["count"], w, h, right)) for right in (False, True)]
    if counts is None:
        counts = [int(s["count"])] + [int(nt) for _, nt in tri]
    n, nl, nr = counts
    meshes = [tri[0][0][:nl], tri[1][0][:nr]]
    prior = done(B.elas_plane_prior(s["list"], meshes[1], w, h, prm, right=True))
    dL, dR = done(B.elas_dense_match(dl, dr, prm, s["list"], n, *meshes, s["grid_L"], s["grid_R"]))
    full = done(B.elas_dense_argmin(dl, dr, prm, prior, s["grid_R"], right=True))
    raw = [dL.clone(), dR.clone()]
    done(B.elas_lr_check(dL, dR, 2, masks=False))
    out = [s["d_can"], s["count"], s["list"][:n], s["grid_L"], s["grid_R"], tri[0][1], tri[1][1], *meshes, prior,
           full, *raw, dL, dR, done(B.elas_postprocess(dL, prm)), done(B.elas_median(dL, 1)),
           done(B.elas_speckle(dL, 1, 20))]
    return out, counts


def test_whole_chains():
    cases = [(*_pair(203 + 64 * k, 117 + 3 * k, k), prm) for k, prm in enumerate((PRM, CENSUS, PRM, CENSUS))]
    alone, counts = [], []
    for L, R, prm in cases:
        out, c = _chain(L, R, prm, stop=True)
        assert min(c) > 50
        alone.append([host(t).copy() for t in out])
        counts.append(c)

    def check(k, out):
        for a, b in zip(out, alone[k]):
            np.testing.assert_array_equal(host(a), b)

    got = [(k % 4, _chain(*cases[k % 4], counts[k % 4])[0]) for k in range(16)]
    torch.cuda.synchronize()
    for k, out in got:
        check(k, out)
    side = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for k in range(16):
        with torch.cuda.stream(side[k % 2]):
            got.append((k % 4, _chain(*cases[k % 4], counts[k % 4])[0]))
    torch.cuda.synchronize()
    for k, out in got:
        check(k, out)
    for k in (0, 1):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side[0]):
            out, _ = _chain(*cases[k], counts[k])
        for _ in range(3):
            g.replay()
        check(k, out)


def test_calls_after_a_replay():
    """A call right behind a graph's replay reads what the graph's last kernel wrote."""
    from paper_1802_07210_gb300 import binding as B
    rng = np.random.default_rng(8)
    maps = [dev(rng.integers(-1, 60, (540, 960)).astype(np.int16)) for _ in range(4)]
    exp = []
    for m in maps:
        mid = B.elas_median(m, 1)
        torch.cuda.synchronize()
        out = B.elas_speckle(mid, 30, 9)
        torch.cuda.synchronize()
        exp.append((host(B.elas_median(out, 1)).copy(), host(B.elas_postprocess(mid, PRM)).copy()))
    s = torch.cuda.Stream()
    src, mid = torch.empty_like(maps[0]), torch.empty_like(maps[0])
    got = []
    with torch.cuda.stream(s):
        src.copy_(maps[0])
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            B.elas_median(src, 1, out=mid)
        for k in range(40):
            src.copy_(maps[k % 4])
            g.replay()
            post = B.elas_postprocess(mid, PRM)
            out = B.elas_median(B.elas_speckle(mid, 30, 9), 1)
            got.append((out, post))
    torch.cuda.synchronize()
    for k, pair in enumerate(got):
        for a, b in zip(pair, exp[k % 4]):
            np.testing.assert_array_equal(host(a), b)
