"""Many pairs on few vertices (each edge given many times): runs of more than 2^18
pairs with more than 768 of them per vertex sort by radix passes, as their
counters are too few to be counted by atomics; others sort by counting.  At both
lines, against the oracle; integer counts: the tolerance is zero."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tc():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_1503_00576_gb300 as lib

    lib.load_library()
    yield lib
    lib.tc_debug_reset()


@pytest.mark.parametrize("n,pairs,crowded", [
    (400, 768 * 400, False), (400, 768 * 400 + 1, True), (400, 3_000_000, True),
    (64, 1 << 18, False), (64, (1 << 18) + 1, True), (2, 300_000, True)])
def test_crowded_runs_sort_by_radix_passes(tc, n, pairs, crowded):
    import torch

    a, b = np.triu_indices(n, 1)
    order = np.random.default_rng(pairs).permutation(pairs) % len(a)
    flip = np.random.default_rng(n).random(pairs) < 0.5
    src = np.where(flip, a[order], b[order]).astype(np.int32)
    dst = np.where(flip, b[order], a[order]).astype(np.int32)
    want = oracle.forward(src, dst, n)
    s, d = torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()

    def launches():
        before = tc.tc_launch_count()
        assert tc.tc_count(s, d, n) == want["T"]
        return tc.tc_launch_count() - before

    as_called = launches()
    T, t, deg = tc.tc_count_per_vertex(s, d, n)
    assert T == want["T"] and np.array_equal(t.cpu().numpy(), want["t"])
    assert np.array_equal(deg.cpu().numpy(), want["deg"])
    assert tc.tc_count_batch(s, d, [0, pairs], [n]).tolist() == [want["T"]]
    tc.tc_debug_set_wait_limit(1 << 24, 1 << 30)  # radix passes, no tile withheld
    try:
        by_radix = launches()
    finally:
        tc.tc_debug_reset()
    assert (as_called == by_radix) == crowded
