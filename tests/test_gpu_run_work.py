"""What the calls' own counting kernels do (tc_debug_run_work) against numpy: the
edges left to an intersection, the entries streamed and hashed, the bitmaps, and
the dense block that the cost model picks, each restated from its rule.

With a withheld radix tile that no call has, every call sorts by radix passes,
so its vertex order is exactly (degree with repeats, at most what the sort's
digits hold, id) and numpy gives every counter; these are also the radix passes' runs on graphs without repeats.
Sorting by counting orders vertices of equal degree class freely: there a graph
whose ties are twins is used, and the rules are checked by bounds.  Integer
counters: the tolerance is zero."""
import numpy as np
import pytest

import graphgen
import oracle
from tests.test_gpu_hub import clique_and_sparse

pytestmark = pytest.mark.gpu

COLUMNS = 4096
NO_TILE = 1 << 30  # a radix tile that no call has


@pytest.fixture(scope="module")
def tc():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_1503_00576_gb300 as lib

    lib.load_library()
    yield lib
    lib.tc_debug_reset()
    lib.tc_set_tuning(None)


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda()


def blocks(x):
    return (x + 7) >> 3


class Lists:
    """The forward lists of the (degree with repeats, id) order, in rank space,
    of the pairs given `times` times: edges (u, v) by owner and entry, i their
    place in N+(u), raw the lists' lengths with repeats."""

    def __init__(self, src, dst, n, times=1):
        s, d = np.asarray(src, np.int64), np.asarray(dst, np.int64)
        keep = s != d
        s, d = s[keep], d[keep]
        digits = (max(1, (n - 1).bit_length()) + 7) // 8
        dord = np.minimum(times * (np.bincount(s, minlength=n) + np.bincount(d, minlength=n)),
                          (1 << 8 * digits) - 1)
        rank = np.empty(n, np.int64)
        rank[np.lexsort((np.arange(n), dord))] = np.arange(n)
        a, b = rank[s], rank[d]
        u, v = np.minimum(a, b), np.maximum(a, b)
        self.n, self.m_raw, self.times = n, times * len(u), times
        self.raw = times * np.bincount(u, minlength=n)
        self.ru, self.rv = u, v  # with repeats
        key = np.unique(u * n + v)
        self.u, self.v = key // n, key % n
        self.len = np.bincount(self.u, minlength=n)
        self.off = np.concatenate([[0], np.cumsum(self.len)])
        self.i = np.arange(len(key)) - self.off[self.u]

    def hub(self, h_max, min_edges, cap, ps):
        """The hub set's size that the cost model picks (0: none)."""
        first = np.concatenate([[0], np.cumsum(self.raw)])
        inside, best, size = 0, 0.0, 0
        low = self.n
        for k in range(4):
            h = h_max * (k + 1) // 4 // 128 * 128
            lo = self.n - h
            owned = (self.ru >= lo) & (self.ru < low)
            inside += self.times * int(np.minimum(np.minimum(self.raw[self.ru[owned]],
                                                self.raw[self.rv[owned]]), cap).sum())
            low = lo
            gain = inside * (1e-9 * ps) - (0.15 + 1.55 * (h / 16384.0) ** 3)
            if self.m_raw - first[lo] >= min_edges and gain > best:
                best, size = gain, h
        return size

    def triangles_among(self, size):
        """Triangles wholly among the `size` highest ranks."""
        lo = self.n - size
        inside = self.u >= lo
        return oracle.forward((self.u[inside] - lo).astype(np.int32),
                              (self.v[inside] - lo).astype(np.int32), size)["T"]

    def work(self, per_vertex, bits, hub=0, emitted=False):
        """partners, lookups, inserts and bitmap pairs; emitted: by the list sort,
        which weighs the other endpoint's list with repeats."""
        u, v, i, n = self.u, self.v, self.i, self.n
        du, dv = self.len[u], (self.raw if emitted else self.len)[v]
        keep = (i + 1 != du) & (dv > 0) & (u < n - hub)
        u, v, i, du, dv = u[keep], v[keep], i[keep], du[keep], dv[keep]
        skip = (i + 1) >> 3
        at_v = 3 * (blocks(du) - skip) < 2 * blocks(dv)
        h, l = np.where(at_v, v, u), np.where(at_v, u, v)
        skip = np.where(at_v, skip, 0)
        size = np.bincount(h, minlength=n)
        least, partners = (12, 64) if per_vertex else (6, 16)
        top = np.bincount(self.u[self.v < max(n - COLUMNS, 0)], minlength=n)
        tb = blocks(top)
        rec = (self.raw > 64) & (blocks(self.len) - tb >= least) if bits else np.zeros(n, bool)
        used = rec[h] & (size[h] >= partners) & rec[l] & \
            (blocks(self.len[l]) - np.maximum(skip, tb[l]) >= least)
        streamed = np.where(used, 8 * tb[l], self.len[l]) - 8 * skip
        return {"partners": len(u), "lookups": int(np.maximum(streamed, 0).sum()),
                "inserts": int(self.len[size > 0].sum()), "bitmap_pairs": int(used.sum())}


def unique_pairs(src, dst, n):
    key = np.unique(np.minimum(src, dst).astype(np.int64) * n + np.maximum(src, dst))
    a, b = key // n, key % n
    keep = a != b
    flip = np.random.default_rng(1).random(keep.sum()) < 0.5
    a, b = a[keep], b[keep]
    return np.where(flip, a, b), np.where(flip, b, a), n


def picked(lists, per_vertex, bits):
    cap, ps = (1 << 31, 0.85) if not bits else (128, 0.85) if per_vertex else (64, 0.6)
    return lists.hub(1 << 14, 1 << 21, cap, ps) if lists.n >= 1 << 17 else 0


GRAPHS = {
    "er": lambda: unique_pairs(*graphgen.er(3000, 60000, 4), 3000),
    "rmat": lambda: unique_pairs(*graphgen.rmat(15, 40 << 15, 6), 1 << 15),
    "rmat_raw": lambda: (*graphgen.rmat(14, 30 << 14, 7), 1 << 14),
    "rgg": lambda: (*graphgen.rgg(1 << 13, graphgen.rgg_radius(1 << 13, 40.0), 6), 1 << 13),
    "hubs": lambda: (*graphgen.rmat(17, 64 << 17, 8), 1 << 17),
    "no_hubs": lambda: (*graphgen.rgg(1 << 17, graphgen.rgg_radius(1 << 17, 40.0), 9), 1 << 17),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_radix_runs_do_the_restated_work(tc, name):
    src, dst, n = GRAPHS[name]()
    lists = Lists(src, dst, n)
    want = oracle.forward(np.asarray(src, np.int32), np.asarray(dst, np.int32), n)
    if name == "hubs":  # the cost model has both answers
        assert picked(lists, False, True) == 0 < picked(lists, True, False)
    s, d = dev(src), dev(dst)
    reps = -(-(1 << 25) // len(src))
    tc.tc_debug_set_wait_limit(1 << 24, NO_TILE)
    try:
        assert tc.tc_count(s, d, n) == want["T"]
        T, t, deg = tc.tc_count_per_vertex(s, d, n)
        assert T == want["T"] and np.array_equal(t.cpu().numpy(), want["t"])
        assert np.array_equal(deg.cpu().numpy(), want["deg"])
        for per_vertex, times in ((False, 1), (True, 1), (True, reps)):
            if times > 1:
                lists = Lists(src, dst, n, times)
            bits = len(src) * times >= (1 << 25 if per_vertex else 1 << 18)
            hub = picked(lists, per_vertex, bits)
            got = tc.tc_debug_run_work(s.repeat(times), d.repeat(times), n, per_vertex)
            assert got["triangles"] == want["T"]
            assert got["dense_vertices"] == hub, (per_vertex, times)
            expect = lists.work(per_vertex, bits, hub)
            assert {k: got[k] for k in expect} == expect, (per_vertex, times)
            if hub and times == 1:
                assert got["dense_triangles"] == lists.triangles_among(hub)
    finally:
        tc.tc_debug_reset()


def threshold_graph(n):
    """i and j joined iff i + j >= n: degrees 1 .. n - 1, the one tie twins."""
    a, b = np.triu_indices(n, 1)
    keep = a + b >= n
    return a[keep], b[keep], n


@pytest.mark.parametrize("n,times", [(9, 1), (64, 1), (250, 1), (127, 2), (60, 4), (28, 9)])
def test_counting_sort_runs_do_the_restated_work(tc, n, times):
    """Repeats too: the split goes by lengths that no warp changes meanwhile, so
    every call's is the same."""
    src, dst, n = threshold_graph(n)
    src, dst = np.tile(src, times), np.tile(dst, times)
    assert (n - 1) * times < 256  # one class per degree
    lists = Lists(src, dst, n)
    T = oracle.forward(np.asarray(src, np.int32), np.asarray(dst, np.int32), n)["T"]
    for per_vertex in (False, True) * 4:
        got = tc.tc_debug_run_work(dev(src), dev(dst), n, per_vertex)
        assert got == {**lists.work(per_vertex, False, emitted=True), "triangles": T,
                       "dense_triangles": 0, "dense_vertices": 0}


def test_dense_block_of_counting_sort_runs(tc):
    """Forced on, the block takes 2^14 vertices, counts at least the triangles
    among the vertices whose degree class lies whole in it, leaves none of its
    edges to an intersection, and with it off the same count comes from them."""
    src, dst, n = clique_and_sparse()
    want = oracle.forward(np.asarray(src, np.int32), np.asarray(dst, np.int32), n)
    s, d = dev(src), dev(dst)
    deg = np.sort(want["deg"])
    sure = int((want["deg"] > deg[n - (1 << 14)]).sum())  # above the class that is cut
    for per_vertex in (False, True):
        try:
            tc.tc_set_tuning({"hub_min_edges": 0})
            on = tc.tc_debug_run_work(s, d, n, per_vertex)
            tc.tc_set_tuning({"hub_min_edges": -1})
            off = tc.tc_debug_run_work(s, d, n, per_vertex)
        finally:
            tc.tc_set_tuning(None)
        assert on["triangles"] == off["triangles"] == want["T"]
        assert on["dense_vertices"] == 1 << 14 and off["dense_vertices"] == 0
        least = Lists(src, dst, n).triangles_among(sure)
        assert least <= on["dense_triangles"] <= want["T"]
        assert off["dense_triangles"] == 0
        # K_200 alone: every list but the last two has an entry to follow
        assert off["partners"] - on["partners"] >= 199 * 198 // 2


def test_cost_model_keeps_it_off_without_hubs(tc):
    src, dst, n = GRAPHS["no_hubs"]()
    for per_vertex in (False, True):
        assert tc.tc_debug_run_work(dev(src), dev(dst), n, per_vertex)["dense_vertices"] == 0
