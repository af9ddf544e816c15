"""The two ways to sort forward lists and partner groups against each other and
the oracle: counting sorts by atomics (csrc/direct.cu; calls of up to
20 * 2^20 pairs) and radix passes (larger calls; shares, which also weigh whole lists).

Graphs at the sizes where the first can go wrong: vertex counts around a tile of
the rank classes, degrees around 256 and far above (the classes coarsen there),
list lengths around every kind of list sort, edges given nine or more times
(lists that shrink to one entry), self-loops, isolated vertices, and hubs that
most edges go to.  The same graphs with their pairs given so often that they
exceed 2^25 take the radix passes.  Integer counts: the tolerance is zero."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tc():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_1503_00576_gb300 as lib

    lib.load_library()
    return lib


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda()


def cliques(sizes, copies, extra):
    """Disjoint cliques (forward lists of every length below each size), each
    pair given `copies` times in alternating directions, a loop at every
    vertex, `extra` isolated vertices; permuted ids."""
    src, dst, base = [], [], 0
    for k in sizes:
        a, b = np.triu_indices(k, 1)
        for c in range(copies):
            src.append(base + (a if c % 2 else b))
            dst.append(base + (b if c % 2 else a))
        base += k
    n = base + extra
    src.append(np.arange(base))
    dst.append(np.arange(base))
    rng = np.random.default_rng(5)
    ids, src, dst = rng.permutation(n), np.concatenate(src), np.concatenate(dst)
    order = rng.permutation(len(src))
    return ids[src[order]], ids[dst[order]], n


def hubs(n, k, links, seed):
    """k hubs, a clique among themselves, and n - k vertices joined to `links`
    of them each."""
    rng = np.random.default_rng(seed)
    a, b = np.triu_indices(k, 1)
    u = np.repeat(np.arange(k, n), links)
    ids = rng.permutation(n)
    return ids[np.concatenate([a, u])], ids[np.concatenate([b, rng.integers(0, k, len(u))])], n


CASES = {
    "one_edge": lambda: (np.array([0]), np.array([1]), 2),
    "tile_less_one": lambda: (*graphgen.er(2047, 20000, 1), 2047),
    "tile": lambda: (*graphgen.er(2048, 20000, 2), 2048),
    "tile_and_one": lambda: (*graphgen.er(2049, 20000, 3), 2049),
    "short_lists": lambda: cliques([2, 3, 8, 9, 10, 16, 17, 18, 32, 33, 34], 1, 7),
    "long_lists": lambda: cliques([64, 65, 66, 128, 129, 256, 257, 258, 512, 513], 1, 100),
    "cta_lists": lambda: cliques([1024, 1026, 1030], 1, 0),
    "nine_copies": lambda: cliques([2, 3, 4, 9, 17, 33, 65, 140], 9, 3),
    "thirty_copies": lambda: cliques([2, 5, 40, 70], 30, 0),
    "rmat_raw": lambda: (*graphgen.rmat(13, 30 << 13, 8), 1 << 13),
    "hubs": lambda: hubs(70000, 40, 12, 9),
    "many_hubs": lambda: hubs(40000, 1400, 3, 10),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_both_sorts_match_the_oracle(tc, name):
    src, dst, n = CASES[name]()
    want = oracle.forward(np.asarray(src, np.int32), np.asarray(dst, np.int32), n)
    s, d = dev(src), dev(dst)
    reps = (1 << 25) // len(src) + 1
    for x, y in ((s, d), (s.repeat(reps), d.repeat(reps))):
        assert tc.tc_count(x, y, n) == want["T"]
        T, t, deg = tc.tc_count_per_vertex(x, y, n)
        assert T == want["T"]
        assert np.array_equal(t.cpu().numpy(), want["t"])
        assert np.array_equal(deg.cpu().numpy(), want["deg"])
    assert sum(tc.tc_count_part(s, d, n, p, 2) for p in range(2)) == want["T"]
    got = tc.tc_count_batch(s.repeat(2), d.repeat(2), [0, len(src), 2 * len(src)], [n, n])
    assert got.tolist() == [want["T"]] * 2
