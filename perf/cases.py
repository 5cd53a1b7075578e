"""The calls a user of this framework makes, as timed cases.

A case is one call (or the few calls that belong together) through the public binding:
whole stereo pairs on device buffers, on host buffers and in batches, and the single steps
that a program composes itself (descriptors and support points, the triangulation, the
dense match, the map filters).  Sizes are those of this repository's workloads (320x240,
640x480, 1242x375, 1280x720, 1920x1080; 64 to 256 disparities) and odd ones between.

Inputs are piecewise-planar scenes like the repository's own synthetic workloads (Voronoi
cells with slanted planes, band-limited texture, forward-warped right image, Gaussian
noise), generated on the GPU from the seed alone.
"""
import math

import numpy as np
import torch

from paper_1802_07210_gb300 import binding as B
from paper_1802_07210_gb300 import synth

CENSUS = dict(census_support_w=9, census_dense_w=5, beta=0.1)
POST = dict(ipol_gap_width=3, filter_adaptive_mean=1)
NO_POST = dict(ipol_gap_width=0, filter_adaptive_mean=0)

# the serving workload's cameras: two 640x480 D=128, four 1242x375 D=256, two 1920x1080 D=256
RIG = "640x480x128,640x480x128,1242x375x256,1242x375x256,1242x375x256,1242x375x256,1920x1080x256,1920x1080x256"


def listed():
    return [
        # the smallest whole pair: a low-resolution robot camera, one pair at a time (latency)
        dict(name="pair_320x240_d64", kind="pair", w=320, h=240, d=64, post=False, census=False, step=5),
        # the headline workload: one VGA pair with post-processing
        dict(name="pair_640x480_d256", kind="pair", w=640, h=480, d=256, post=True, census=False, step=5),
        # the paper's census variant on a driving camera's shape
        dict(name="pair_census_1242x375_d256", kind="pair", w=1242, h=375, d=256, post=False, census=True, step=5),
        # the largest single pair: full HD
        dict(name="pair_1920x1080_d256", kind="pair", w=1920, h=1080, d=256, post=True, census=False, step=5),
        # an odd size through the host-buffer call: frames arrive in pinned host memory and leave there
        dict(name="host_1011x613_d128", kind="host", w=1011, h=613, d=128, post=True, census=False, step=5),
        # eight cameras of three shapes in one wave, with post-processing
        dict(name="batch_rig_8", kind="batch", shapes=RIG, post=True, census=False, step=5),
        # many small pairs in one wave (thumbnails of a camera array, odd size)
        dict(name="batch_24x317x241_d64", kind="batch", shapes=",".join(["317x241x64"] * 24), post=False,
             census=False, step=5),
        # the offline throughput workload: 64 driving pairs in one wave
        dict(name="batch_64x1242x375_d256", kind="batch", shapes=",".join(["1242x375x256"] * 64), post=False,
             census=False, step=5),
        # a program's own composition: descriptors and support points of an odd-sized pair
        dict(name="support_1013x547_d200", kind="support", w=1013, h=547, d=200, post=False, census=False, step=5),
        # both meshes of one driving pair, triangulated on the device
        dict(name="triangulate_1242x375", kind="triangulate", w=1242, h=375, d=256, post=False, census=False, step=5),
        # plane prior and dense argmin of both images of a 720p pair
        dict(name="dense_1280x720_d128", kind="dense", w=1280, h=720, d=128, post=False, census=False, step=5),
        # cleaning a full-HD disparity map: gap interpolation and adaptive mean, median, speckle removal
        dict(name="filters_1920x1080", kind="filters", w=1920, h=1080, d=256, post=True, census=False, step=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "host", "batch", "batch", "support", "triangulate", "dense", "filters"])
    # down to QVGA height in both directions, up to full HD
    w, h = _log_int(rng, 240, 1920), _log_int(rng, 160, 1080)
    d = _log_int(rng, 32, max(33, min(256, w // 4)))
    census = kind in ("pair", "batch", "support", "dense") and rng.random() < 0.25
    post = rng.random() < 0.5 or kind == "filters"
    step = rng.choice([5, 5, 5, 4, 7])  # the candidate lattice's spacing
    if kind != "batch":
        return dict(kind=kind, w=w, h=h, d=d, post=post, census=census, step=step)
    # up to 40 pairs of one to three shapes, well below the largest listed batch's pixels
    shapes, pixels = [(w, h, d)], 0
    for _ in range(rng.randrange(3)):
        w2, h2 = _log_int(rng, 240, 1280), _log_int(rng, 160, 720)
        shapes.append((w2, h2, _log_int(rng, 32, max(33, min(256, w2 // 4)))))
    picked = []
    for _ in range(_log_int(rng, 2, 40)):
        s = rng.choice(shapes)
        if picked and pixels + s[0] * s[1] > 12_000_000:
            break
        picked.append(s)
        pixels += s[0] * s[1]
    return dict(kind=kind, shapes=",".join("%dx%dx%d" % s for s in picked), post=post, census=census, step=5)


# ---- inputs -------------------------------------------------------------------

def _box3(a):
    p = torch.nn.functional.pad(a[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
    h, w = a.shape
    s = sum(p[dy:dy + h, dx:dx + w] for dy in range(3) for dx in range(3))
    return torch.floor((s + 4) / 9)


def _scene(w, h, d, gen):
    """A piecewise-planar scene on the GPU: left and right uint8 images, the left image's
    disparities and the mask of its pixels that the right image shows."""
    dev = gen.device

    def uniform(n, lo, hi):
        return torch.rand(n, generator=gen, device=dev) * (hi - lo) + lo

    k = max(6, min(60, round(20 * w * h / 307200)))
    sx, sy = uniform(k, 0, w), uniform(k, 0, h)
    dc, a, b = uniform(k, 0, 0.98 * (d - 1)), uniform(k, -0.12, 0.12), uniform(k, -0.12, 0.12)
    uu = torch.arange(w, device=dev, dtype=torch.float32)[None, :]
    vv = torch.arange(h, device=dev, dtype=torch.float32)[:, None]
    best = torch.full((h, w), 1e30, device=dev)
    disp = torch.zeros((h, w), device=dev)
    for i in range(k):
        r = (uu - sx[i]) ** 2 + (vv - sy[i]) ** 2
        near = r < best
        best = torch.where(near, r, best)
        disp = torch.where(near, dc[i] + a[i] * (uu - sx[i]) + b[i] * (vv - sy[i]), disp)
    if w > 3 * h:  # a driving camera's ground plane, rising 0 to 120 from top to bottom
        disp = torch.maximum(disp, min(120.0, 0.5 * d) * vv / (h - 1))
    disp = torch.round(disp.clamp(0, 0.98 * (d - 1))).to(torch.int64)

    def texture():
        return _box3(torch.randint(0, 256, (h, w), generator=gen, device=dev).float())

    left, fill = texture(), texture()
    # forward warp: the larger disparity wins, then the larger column
    u = torch.arange(w, device=dev)[None, :].expand(h, w)
    x = u - disp
    ok = x >= 0
    dst = (torch.arange(h, device=dev)[:, None] * w + x)[ok]
    key = torch.full((h * w,), -1, dtype=torch.int64, device=dev)
    key.scatter_reduce_(0, dst, (disp * w + u)[ok], "amax")
    key = key.view(h, w)
    right = torch.where(key >= 0, torch.gather(left, 1, key.clamp(min=0) % w), fill)

    def noisy(img):
        sigma = 3.0 if w > 3 * h else 2.0
        noise = torch.randn((h, w), generator=gen, device=dev) * sigma
        return torch.round(img + noise).clamp(0, 255).to(torch.uint8)

    shown = ok & (torch.gather(key, 1, x.clamp(min=0)) == disp * w + u)
    return noisy(left), noisy(right), disp, shown


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return gen


def _params(case, d):
    prm = dict(synth.ROBOTICS, disp_min=0, disp_max=d - 1, candidate_stepsize=case["step"])
    prm.update(POST if case["post"] else NO_POST)
    if case["census"]:
        prm.update(CENSUS)
    return prm


def _shapes(case):
    return [tuple(int(x) for x in s.split("x")) for s in case["shapes"].split(",")]


def _filters_map(case, seed):
    """A disparity map as a left-right check leaves it: the scene's disparities with errors of
    a pixel, some wrong patches, and -1 where the match is outside the image or occluded and at
    scattered pixels."""
    w, h, d = case["w"], case["h"], case["d"]
    gen = _generator(seed)
    _, _, disp, visible = _scene(w, h, d, gen)

    def rand(hh, ww):
        return torch.rand((hh, ww), generator=gen, device="cuda")

    def patches(share):  # 4x4 pixel patches
        p = rand((h + 3) // 4, (w + 3) // 4) < share
        return p.repeat_interleave(4, 0).repeat_interleave(4, 1)[:h, :w]

    noise = rand(h, w)
    disp = disp + (noise < 0.1).long() - (noise > 0.9).long()
    disp = torch.where(patches(0.01), (rand(h, w) * d).long(), disp)
    invalid = ~visible | patches(0.02) | (rand(h, w) < 0.04)
    return torch.where(invalid, torch.full_like(disp, -1), disp.clamp(0, d - 1)).to(torch.int16).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind)
    if kind == "batch":
        shapes = _shapes(case)
        gen = _generator(seed)
        pairs = [_scene(w, h, d, gen)[:2] for w, h, d in shapes]
        st["L"], st["R"] = [p[0] for p in pairs], [p[1] for p in pairs]
        st["dL"] = [torch.empty((h, w), dtype=torch.int16, device="cuda") for w, h, _ in shapes]
        st["post"] = [torch.empty((h, w), dtype=torch.float32, device="cuda")
                      for w, h, _ in shapes] if case["post"] else None
        st["batch"] = B.Batch([(w, h) for w, h, _ in shapes], [_params(case, d) for _, _, d in shapes])
        return st
    if kind == "filters":
        st["map"], st["prm"] = _filters_map(case, seed), B.as_params(_params(case, case["d"]))
        return st
    w, h, d = case["w"], case["h"], case["d"]
    prm = B.as_params(_params(case, d))
    L, R = _scene(w, h, d, _generator(seed))[:2]
    st.update(w=w, h=h, prm=prm, census=case["census"], L=L, R=R)
    if kind in ("pair", "host"):
        host = kind == "host"
        where = dict(device="cpu", pin_memory=True) if host else dict(device="cuda")
        if host:
            st["L"], st["R"] = L.cpu().pin_memory(), R.cpu().pin_memory()
        st["dL"] = torch.empty((h, w), dtype=torch.int16, **where)
        st["dR"] = torch.empty((h, w), dtype=torch.int16, **where)
        st["post"] = torch.empty((h, w), dtype=torch.float32, **where) if case["post"] else None
        st["pipe"] = B.Pipeline(w, h, prm)
        return st
    sup = _support(st)
    n = int(sup["count"])  # the program reads the count between the steps
    st["n"] = n
    if kind == "support":
        st["keep"] = torch.zeros_like(sup["list"])
        return st
    st["list"] = sup["list"][:n].contiguous()
    st["count"] = sup["count"]
    st["tri"], st["keep"] = [], []
    cap = (w // prm.candidate_stepsize) * (h // prm.candidate_stepsize)
    for right in (False, True):
        tri, nt = B.elas_triangulate_device(st["list"], st["count"], w, h, right)
        st["tri"].append(tri[:int(nt)].contiguous())
        st["keep"].append(torch.zeros((2 * cap, 3), dtype=torch.int32, device="cuda"))
    if kind == "dense":
        if case["census"]:
            st["descL"], st["descR"] = B.elas_census(L, R, prm.census_dense_w, 16)
        else:
            st["descL"], st["descR"] = B.elas_descriptors(L, R)
        st["grid_L"], st["grid_R"] = sup["grid_L"], sup["grid_R"]
    return st


def _support(st):
    if st["census"]:
        descL, descR = B.elas_census(st["L"], st["R"], st["prm"].census_support_w, 32)
    else:
        descL, descR = B.elas_descriptors(st["L"], st["R"])
    out = B.elas_support_points(descL, descR, st["prm"])
    out["descL"], out["descR"] = descL, descR
    return out


def run(state):
    kind = state["kind"]
    if kind == "pair":
        state["pipe"].run(state["L"], state["R"], state["dL"], state["dR"], state["post"])
    elif kind == "host":
        state["pipe"].run_host(state["L"], state["R"], state["dL"], state["dR"], state["post"])
    if kind in ("pair", "host"):
        return [t for t in (state["dL"], state["dR"], state["post"]) if t is not None]
    if kind == "batch":
        state["batch"].run(state["L"], state["R"], state["dL"], None, state["post"])
        return state["dL"] + (state["post"] or [])
    if kind == "support":
        s = _support(state)
        # the program keeps the points in a buffer of the full capacity (the list's rows past the
        # count are not written)
        state["keep"][:state["n"]].copy_(s["list"][:state["n"]])
        return [s["descL"], s["descR"], s["d_can"], state["keep"], s["count"], s["grid_L"], s["grid_R"]]
    if kind == "triangulate":
        out = []
        for right in (False, True):
            tri, nt = B.elas_triangulate_device(state["list"], state["count"], state["w"], state["h"], right)
            # kept in a buffer of the full capacity (rows past the count are not written)
            nt_host = len(state["tri"][right])
            state["keep"][right][:nt_host].copy_(tri[:nt_host])
            out += [state["keep"][right], nt]
        return out
    if kind == "dense":
        return list(B.elas_dense_match(state["descL"], state["descR"], state["prm"], state["list"], state["n"],
                                       state["tri"][0], state["tri"][1], state["grid_L"], state["grid_R"]))
    post = B.elas_postprocess(state["map"], state["prm"])
    return [post, B.elas_median(state["map"], 1), B.elas_speckle(state["map"], 1, 200)]


# ---- what the path cannot do without ---------------------------------------------

def _pair_work(w, h, d, step, post, right):
    px = w * h
    cand = (w // step) * (h // step)
    return dict(bytes=2 * px + 2 * px * (2 if right else 1) + (4 * px if post else 0),
                # the 64-byte window differences and sums of every candidate and disparity, once,
                # and about ten 16-byte ones per pixel and image in the dense match
                flops=cand * d * 128 + 2 * px * 10 * 32)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [_pair_work(w, h, d, case["step"], case["post"], False) for w, h, d in _shapes(case)]
        return dict(bytes=sum(p["bytes"] for p in parts), flops=sum(p["flops"] for p in parts))
    w, h, d, step = case["w"], case["h"], case["d"], case["step"]
    px, cand = w * h, (w // step) * (h // step)
    if kind in ("pair", "host"):
        return _pair_work(w, h, d, step, case["post"], True)
    if kind == "support":
        rec = 32 if case["census"] else 16
        return dict(bytes=2 * px + 2 * px * rec + 2 * cand, flops=cand * d * 128)
    if kind == "triangulate":
        # both meshes: about 0.4 of the candidates are support points, two triangles each
        n = int(0.4 * cand)
        return dict(bytes=2 * (6 * n + 12 * 2 * n), flops=2 * 2 * n * 60)
    if kind == "dense":
        return dict(bytes=2 * px * 16 + 2 * px * 2, flops=2 * px * 10 * 32)
    return dict(bytes=3 * 2 * px + 4 * px + 2 * 2 * px, flops=px * 2 * 7 * 4)


# ---- the computed map in 64 bits -------------------------------------------------

def _gap_rows(d, gap):
    """Fills invalid runs of at most `gap` pixels between two valid ones, per row."""
    out = d.copy()
    h, w = d.shape
    col = np.arange(w)[None, :]
    valid = d >= 0
    left = np.maximum.accumulate(np.where(valid, col, -1), axis=1)
    right = np.minimum.accumulate(np.where(valid, col, w)[:, ::-1], axis=1)[:, ::-1]
    fill = ~valid & (left >= 0) & (right < w) & (right - left - 1 <= gap)
    rows, cols = np.nonzero(fill)
    d1, d2 = d[rows, left[rows, cols]], d[rows, right[rows, cols]]
    out[rows, cols] = np.where(np.abs(d1 - d2) < 3, (d1 + d2) / 2, np.minimum(d1, d2))
    return out


def _mean_rows(d):
    """Mean of the valid values at offsets -3..3 weighted by max(0, 4 - |difference|)."""
    h, w = d.shape
    num, den = np.zeros_like(d), np.zeros_like(d)
    for o in range(-3, 4):
        shifted = np.full_like(d, -1.0)
        shifted[:, max(0, -o):w - max(0, o)] = d[:, max(0, o):w - max(0, -o)]
        weight = np.where((shifted >= 0) & (d >= 0), np.maximum(0.0, 4.0 - np.abs(shifted - d)), 0.0)
        num += weight * shifted
        den += weight
    return np.where((d >= 0) & (den > 0), num / np.where(den > 0, den, 1.0), d)


def exact(case, seed):
    """The post-processed map in 64 bits; the other outputs are whole numbers."""
    if case["kind"] != "filters":
        return None
    d = _filters_map(case, seed).cpu().numpy().astype(np.float64)
    d = _gap_rows(d, POST["ipol_gap_width"])
    d = np.ascontiguousarray(_gap_rows(np.ascontiguousarray(d.T), POST["ipol_gap_width"]).T)
    d = _mean_rows(d)
    d = np.ascontiguousarray(_mean_rows(np.ascontiguousarray(d.T)).T)
    return [d, None, None]
