"""Per-vertex counts short of device memory: a call whose workspace with the
bitmaps or the partners' streams does not fit runs without them, in the memory
that a call without per-vertex counts takes, and only when that does not fit
either it reports TC_ERR_OOM.  Sizes on every path: the counting sorts with
streams, the radix passes with bitmaps, those without (there is nothing to do
without: the first failure is the call's); and shares.  Integer counts: the
tolerance is zero."""
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
    yield lib
    lib.tc_debug_reset()


def graph(pairs):
    """An R-MAT graph, its pairs given until there are `pairs` of them."""
    import torch

    scale = 10 if pairs < 1 << 20 else 17
    src, dst = graphgen.rmat(scale, 4 << scale if pairs < 1 << 20 else 1 << 20, 3)
    n = 1 << scale
    reps = -(-pairs // len(src))
    s, d = (torch.from_numpy(x).cuda().repeat(reps)[:pairs] for x in (src, dst))
    return s, d, n, oracle.forward(src, dst, n)


@pytest.mark.parametrize("pairs", [1 << 12, 1 << 22, 1 << 25])
def test_a_failed_allocation_is_tried_without_the_extras(tc, pairs):
    s, d, n, want = graph(pairs)
    try:
        for parts in (1, 2):
            t_sum = np.zeros(n, np.int64)
            for part in range(parts):
                tc.tc_debug_fail_allocations(0, 1)
                T, t, deg = (tc.tc_count_per_vertex(s, d, n) if parts == 1 else
                             tc.tc_count_per_vertex_part(s, d, n, part, parts))
                t_sum += t.cpu().numpy()
                assert np.array_equal(deg.cpu().numpy(), want["deg"])
            assert np.array_equal(t_sum, want["t"])
        tc.tc_debug_fail_allocations(0, 2)
        with pytest.raises(tc.TCError) as ei:
            tc.tc_count_per_vertex(s, d, n)
        assert ei.value.code == tc.TC_ERR_OOM
    finally:
        tc.tc_debug_fail_allocations(0, 0)
    T, t, deg = tc.tc_count_per_vertex(s, d, n)
    assert T == want["T"] and np.array_equal(t.cpu().numpy(), want["t"])


def test_without_extras_the_first_failure_is_reported(tc):
    s, d, n, want = graph((20 << 20) + 1)
    tc.tc_debug_fail_allocations(0, 1)
    try:
        with pytest.raises(tc.TCError) as ei:
            tc.tc_count_per_vertex(s, d, n)
        assert ei.value.code == tc.TC_ERR_OOM
    finally:
        tc.tc_debug_fail_allocations(0, 0)
    T, t, deg = tc.tc_count_per_vertex(s, d, n)
    assert T == want["T"] and np.array_equal(t.cpu().numpy(), want["t"])
