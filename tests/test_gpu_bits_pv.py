"""Per-vertex counts by bitmaps (csrc/bits.cu, runs of at least 2^25 pairs) where
the groups are dealt to shares, and with ids of more than 24 bits (every partner's
list is streamed whole).  Against the oracle; integer counts: the tolerance is
zero."""
import numpy as np
import pytest

import graphgen
import oracle
from tests.test_gpu_bits import core_and_rest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tc():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_1503_00576_gb300 as lib

    lib.load_library()
    return lib


def repeated(src, dst):
    """The pairs on the device, given until there are 2^25."""
    import torch

    reps = -(-(1 << 25) // len(src))
    return (torch.from_numpy(np.ascontiguousarray(x, np.int32)).cuda().repeat(reps)
            for x in (src, dst))


@pytest.mark.parametrize("parts", [2, 5])
def test_shares(tc, parts):
    src, dst = graphgen.rmat(15, 40 << 15, 6)
    n = 1 << 15
    want = oracle.forward(src, dst, n)
    s, d = repeated(src, dst)
    assert tc.tc_debug_run_work(s, d, n, True)["bitmap_pairs"] > 0
    total, t_sum = 0, np.zeros(n, np.int64)
    for part in range(parts):
        T, t, deg = tc.tc_count_per_vertex_part(s, d, n, part, parts)
        total += T
        t_sum += t.cpu().numpy()
        assert np.array_equal(deg.cpu().numpy(), want["deg"])
    assert total == want["T"] and np.array_equal(t_sum, want["t"])


def test_wide_ids(tc):
    src, dst, used = core_and_rest(1000, 3000, 80, 2)
    n = (1 << 24) + 3
    ids = np.random.default_rng(3).choice(n, used, replace=False)
    want = oracle.forward(np.asarray(src, np.int32), np.asarray(dst, np.int32), used)
    s, d = repeated(ids[src], ids[dst])
    assert tc.tc_debug_run_work(s, d, n, True)["bitmap_pairs"] > 0
    T, t, deg = tc.tc_count_per_vertex(s, d, n)
    t, deg = t.cpu().numpy(), deg.cpu().numpy()
    assert T == want["T"] == t.sum() // 3
    assert np.array_equal(t[ids], want["t"]) and np.array_equal(deg[ids], want["deg"])
    assert int(deg.sum()) == int(want["deg"].sum())
