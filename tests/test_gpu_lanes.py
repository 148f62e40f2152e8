"""The one-lane kernel's warps against the register-list kernel, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from paper_2605_02224_gb300 import Cloud
from paper_2605_02224_gb300 import mknn as M
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cloud():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P, _ = W.torus(3000, 71)
    order = W.permutation(3000, 72)
    c = Cloud.build(P, order).upload()
    yield c, P[order]
    c.close()


# k at the edges of each list kind (8, 16, 32, 64 slots)
@pytest.mark.parametrize("k", [1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 48, 49, 64])
def test_partial_warps_and_bounds(cloud, k):
    """Warps with 1, 31 and 32 queries, queries on sites, bounds that leave
    fewer than k sites, rows that end at an odd or even entry, and bounds out
    of [1, n]: the plain launch and a plan give the register kernel's rows,
    and the padded rows of invalid bounds."""
    import torch
    c, P = cloud
    for nq in (1, 31, 32, 33, 289):
        Q = np.concatenate([W.box_queries(nq, 73 + nq, [-1.6] * 3, [1.6] * 3), P[:nq]])[:nq + nq // 2]
        rng = np.random.default_rng(nq)
        m = rng.integers(1, 3001, Q.shape[0]).astype(np.int32)
        m[::5] = rng.integers(1, 2 * k + 2, m[::5].size)
        bad = np.zeros(m.size, bool)
        bad[3::29] = True
        m[bad] = np.where(np.arange(bad.sum()) % 2 == 0, 0, 3001)
        q, mt = torch.from_numpy(Q).cuda(), torch.from_numpy(m).cuda()
        want = c.knn(q, k, mt, lanes=1, placement=1)
        got = c.knn(q, k, mt, lanes=1, placement=2)
        idx = torch.empty_like(want[0])
        d2 = torch.empty_like(want[1])
        M.mknn_knn_batch([dict(cloud=c.handle, q=q, nq=q.shape[0], k=k, m=mt, out_idx=idx,
                               out_d2=d2)], lanes=1, item_rounds=2)
        torch.cuda.synchronize()
        for i, d in (got, (idx, d2)):
            assert torch.equal(i, want[0]) and torch.equal(d, want[1])
        assert np.all(got[0].cpu().numpy()[bad] == -1)
        assert c.check() == (1 if bad.any() else 0)
        good = np.nonzero(~bad)[0][:40]
        parity.check_rows(P, Q[good], k, m[good], got[0].cpu().numpy()[good],
                          got[1].cpu().numpy()[good])


@pytest.mark.parametrize("surface,n", [("torus", 4000), ("patches", 12000),
                                       ("patches", 30000), ("patches", 90000)])
@pytest.mark.parametrize("k", [1, 16, 32, 47, 48, 100])
def test_default_lanes_around_the_crossover(surface, n, k):
    """Launches just below and above the number of queries from which one
    lane per query is the default, on clouds without long lists, with them,
    and with box trees: the plain launch, the no-allocation one and a plan
    give the rows of one lane and of one warp per query."""
    import torch
    P, _ = W.surface(surface, n, 81)
    order = W.permutation(n, 82)
    c = Cloud.build(P, order).upload()
    lo, hi = W.padded_box(P)
    base = 40960 + 1100 * k
    for nq in (base - 1, base, base + 81919, base + 81920):
        q = torch.from_numpy(W.box_queries(nq, 83, lo, hi)).cuda()
        want = c.knn(q, k, lanes=32, placement=1)
        runs = [c.knn(q, k), c.knn(q, k, lanes=1, placement=2)]
        for call in (lambda i, d: M.mknn_knn_noalloc(c.handle, q, nq, 3, k, None, 0, i, d),
                     lambda i, d: M.mknn_knn_batch([dict(cloud=c.handle, q=q, nq=nq, k=k,
                                                         out_idx=i, out_d2=d)])):
            idx, d2 = torch.full_like(want[0], -9), torch.full_like(want[1], -9)
            call(idx, d2)
            runs.append((idx, d2))
        torch.cuda.synchronize()
        for i, d in runs:
            assert torch.equal(i, want[0]) and torch.equal(d, want[1])
    c.close()


@pytest.mark.parametrize("k", [1, 2, 3, 17, 31, 32, 33, 64, 65, 128])
def test_one_warp_lists(k):
    """New keys merged in one pass, on clouds where lists share entries and
    keys tie: a lattice (whole rings at one distance),
    duplicated points, patches with box trees, and clouds of fewer sites than
    k; queries on sites, at cell centres and in the box, bounds from 1 up.
    The rows are the register kernel's, and the oracle's."""
    import torch
    L, _ = W.lattice(9)
    S, _ = W.sphere(300, 91)
    P, _ = W.patches4(30000, 92)
    for pts in (L, np.concatenate([S, S, S[:100]]), P, S[:5], S[:40]):
        n = len(pts)
        order = W.permutation(n, 93)
        c = Cloud.build(pts, order).upload()
        lo, hi = W.padded_box(pts)
        Q = np.concatenate([W.box_queries(150, 94, lo, hi), pts[:: max(1, n // 150)][:150],
                            (pts[:50] + np.float32(0.5))]).astype(np.float32)
        m = np.random.default_rng(95).integers(1, n + 1, len(Q)).astype(np.int32)
        m[::3] = n
        q, mt = torch.from_numpy(Q).cuda(), torch.from_numpy(m).cuda()
        lanes = 32 if k <= 64 else 16
        want = c.knn(q, k, mt, lanes=lanes, placement=1)
        got = c.knn(q, k, mt, lanes=32, placement=2)
        torch.cuda.synchronize()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]), (n, k)
        parity.check_rows(pts[order], Q, k, m, got[0].cpu().numpy(), got[1].cpu().numpy(),
                          rows=range(0, len(Q), 11))
        c.close()


@pytest.mark.parametrize("nq", [1, 33, 1023, 4096, 16383, 16384, 16385])
@pytest.mark.parametrize("shape", ["box", "one", "line", "odd"])
def test_sorted_rows_equal_unsorted(cloud, nq, shape):
    """The one-block sort and the five-kernel one around the line between
    them: every query's row is written, and is the unsorted launch's, for
    queries in a box, all at one point, on a line, and with coordinates that
    are not finite."""
    import torch
    c, _ = cloud
    Q = W.box_queries(nq, 74, [-1.6] * 3, [1.6] * 3)
    if shape == "one":
        Q[:] = Q[0]
    elif shape == "line":
        Q[:, 1:] = Q[0, 1:]
    elif shape == "odd":
        Q[::3, 0] = np.nan
        Q[1::5, 1] = np.inf
        Q[2::7, 2] = -np.inf
    q = torch.from_numpy(Q).cuda()
    q4 = torch.cat([q, q[:, :1]], 1).contiguous()
    want = c.knn(q, 4, sort=-1)
    idx, d2 = torch.full_like(want[0], -9), torch.full_like(want[1], -9)
    M.mknn_knn_noalloc(c.handle, q, nq, 3, 4, None, 0, idx, d2)
    for got in (c.knn(q4, 4, sort=1), (idx, d2)):
        torch.cuda.synchronize()
        assert torch.equal(got[0], want[0])
        assert torch.equal(got[1].view(torch.int32), want[1].view(torch.int32))
