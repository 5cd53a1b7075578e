"""Calls from several host threads at once, each on its own stream, whose
launches need different amounts of shared memory from the same kernel: the
limit that a launch needs is not another thread's to lower."""
import threading

import numpy as np
import pytest

import oracle
from tests.gpu_util import dev, host, require_gpu, torch

pytestmark = pytest.mark.gpu

CALLS = 1500


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _in_threads(jobs):
    """Runs each job(stream) CALLS times in a thread of its own; the results of the last calls."""
    out, errors = [None] * len(jobs), []
    start = threading.Barrier(len(jobs))

    def work(i):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                start.wait()
                for _ in range(CALLS):
                    out[i] = jobs[i](s)
                s.synchronize()
        except Exception as e:  # reported by the test's thread
            errors.append("%d: %s" % (i, e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    return out


def test_triangulations_of_different_heights():
    from paper_1802_07210_gb300 import binding as B
    rng = np.random.default_rng(2)
    jobs, exp = [], []
    for h in (16, 16383, 40, 9000):
        pts = np.unique(np.stack([rng.integers(0, h, 30), rng.integers(0, 60, 30)], 1), axis=0)
        lst = np.concatenate([pts[:, ::-1], np.full((len(pts), 1), 2)], 1).astype(np.int16)
        l, c = dev(lst), dev(np.array([len(lst)], np.int32))
        torch.cuda.synchronize()
        jobs.append(lambda s, l=l, c=c, h=h: B.elas_triangulate_device(l, c, 64, h, stream=s))
        exp.append(len(oracle.triangulate(lst)))
    for (tri, nt), n in zip(_in_threads(jobs), exp):
        assert int(host(nt)[0]) == n


def test_lr_checks_of_different_widths():
    """In place and again: the maps end where the check takes nothing more away."""
    from paper_1802_07210_gb300 import binding as B
    jobs, maps, exp = [], [], []
    for w in (12301, 16383, 12800, 14000):  # all above 48 KB of rows
        rng = np.random.default_rng(w)
        l, r = (rng.integers(-1, 6, (2, w)).astype(np.int16) for _ in range(2))
        a, b = dev(l), dev(r)
        torch.cuda.synchronize()
        jobs.append(lambda s, a=a, b=b: B.elas_lr_check(a, b, 1, masks=False, stream=s))
        maps.append((a, b))
        for _ in range(CALLS):
            l2, r2 = oracle.lr_check(l, r, 1)[:2]
            if (l2 == l).all() and (r2 == r).all():
                break
            l, r = l2, r2
        exp.append((l, r))
    _in_threads(jobs)
    for (a, b), (l, r) in zip(maps, exp):
        np.testing.assert_array_equal(host(a), l)
        np.testing.assert_array_equal(host(b), r)


def test_redundancy_distances_of_different_lengths():
    """50 to 96 KB of staged rows in the redundancy filter."""
    from paper_1802_07210_gb300 import binding as B
    rng = np.random.default_rng(5)
    img = rng.integers(0, 256, (90, 300)).astype(np.uint8)
    dl, dr = oracle.descriptors(img), oracle.descriptors(np.roll(img, -7, 1))
    L, R = dev(dl), dev(dr)
    torch.cuda.synchronize()
    jobs, exp = [], []
    for maxd in (400, 300, 250, 210):
        prm = dict(disp_max=31, candidate_stepsize=5, redun_max_dist=maxd)
        jobs.append(lambda s, prm=prm: B.elas_support_points(L, R, prm, stream=s)["d_can"])
        exp.append(oracle.support_points(dl, dr, prm))
    for got, want in zip(_in_threads(jobs), exp):
        np.testing.assert_array_equal(host(got), want)
