"""Intersections by bitmaps of the top ranks (csrc/bits.cu) against the oracle.

Graphs of at least 2^18 pairs (T) and 2^25 pairs (per vertex; the same graph
with its pairs given several times), where the bitmaps are used, at the sizes
where they can go wrong: fewer vertices than columns, as many, one more,
lists that end on either side of a 32-byte block, lists whose top ranks begin
inside a block, hubs shared by thousands of partners (work items of 128 and
248 partners), repeats, and shares.  Integer counts: the tolerance is zero."""
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


def core_and_rest(core, rest, links, seed):
    """A random core of density 1/2 on `core` vertices and `rest` vertices
    joined to `links` of them each; permuted ids."""
    rng = np.random.default_rng(seed)
    a, b = np.triu_indices(core, 1)
    keep = rng.random(len(a)) < 0.5
    a, b = a[keep], b[keep]
    u = np.repeat(np.arange(core, core + rest), links)
    v = rng.integers(0, core, rest * links)
    n = core + rest
    ids = rng.permutation(n)
    return ids[np.concatenate([a, u])], ids[np.concatenate([b, v])], n


def both(src, dst, n):
    return np.concatenate([src, dst]), np.concatenate([dst, src]), n


CASES = {
    # K_n: every list a run of ranks, every list length from 0 to n - 1
    "k733": lambda: (*(x for x in np.triu_indices(733, 1)), 733),
    "core_below_columns": lambda: core_and_rest(900, 3000, 70, 1),
    "core_at_columns": lambda: core_and_rest(1000, 4096 - 1000, 80, 2),
    "core_past_columns": lambda: core_and_rest(1000, 4097 - 1000, 64, 3),
    # lists of about 250 entries, a third of the ranks in the columns
    "straddle": lambda: (*graphgen.er(12000, 3_000_000, 5), 12000),
    "rmat": lambda: (*graphgen.rmat(15, 40 << 15, 6), 1 << 15),
    "both_directions": lambda: both(*graphgen.rmat(14, 30 << 14, 7), 1 << 14),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_bitmaps_match_the_oracle(tc, name):
    src, dst, n = CASES[name]()
    assert len(src) >= 1 << 18
    want = oracle.forward(np.asarray(src, np.int32), np.asarray(dst, np.int32), n)
    s, d = dev(src), dev(dst)
    assert tc.tc_count(s, d, n) == want["T"]
    reps = -(-(1 << 25) // len(src))
    T, t, deg = tc.tc_count_per_vertex(s.repeat(reps), d.repeat(reps), n)
    assert T == want["T"]
    assert np.array_equal(t.cpu().numpy(), want["t"])
    assert np.array_equal(deg.cpu().numpy(), want["deg"])
    shares = [tc.tc_count_part(s, d, n, p, 3) for p in range(3)]
    assert sum(shares) == want["T"]
