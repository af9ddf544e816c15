"""Failure paths of the calls that sort by counting (csrc/direct.cu): the offset
scans are their only waits.  A test hook (include/tc_debug.h) makes one tile of
the scan of the forward lists, or of the partner groups, never publish, so the
tiles after it wait on a word that nothing sets until their (lowered) limit runs
out.  The call must return TC_ERR_TIMEOUT, no kernel may run on the incomplete
node arrays, and the next call, with the defaults back, must count exactly.  The
expected counts come from the CPU oracle."""
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


@pytest.fixture(scope="module")
def graph():
    """R-MAT scale 18, 4.2M pairs: 65 scan tiles of 4096 vertices, lists with
    bitmaps, and a layout with the dense block."""
    import torch

    src, dst = graphgen.rmat(18, 16 << 18, 31)
    n = 1 << 18
    return torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), n, \
        oracle.forward(src, dst, n)


def expect_timeout(tc, fn, *a, **k):
    with pytest.raises(tc.TCError) as ei:
        fn(*a, **k)
    assert ei.value.code == tc.TC_ERR_TIMEOUT, ei.value


@pytest.mark.parametrize("scan", [0, 1])
@pytest.mark.parametrize("tile", [0, 3, 63])
def test_a_scan_that_waits_in_vain_times_out(tc, graph, scan, tile):
    import torch

    s, d, n, want = graph
    tc.tc_debug_set_wait_limit(2000)
    tc.tc_debug_set_unpublished_scan(scan, tile)
    try:
        expect_timeout(tc, tc.tc_count, s, d, n)
        t = torch.full((n,), -7, dtype=torch.int64, device="cuda")
        expect_timeout(tc, tc.tc_count_per_vertex, s, d, n, t_out=t)
        # nothing downstream ran: the per-vertex output was never written
        assert bool((t == -7).all().item())
    finally:
        tc.tc_debug_reset()
    torch.cuda.synchronize()  # the context is intact
    assert tc.tc_count(s, d, n) == want["T"]
    T, t, deg = tc.tc_count_per_vertex(s, d, n)
    assert T == want["T"] and np.array_equal(t.cpu().numpy(), want["t"])
    assert np.array_equal(deg.cpu().numpy(), want["deg"])


@pytest.mark.parametrize("scan", [0, 1])
def test_batch_and_engine_time_out_then_recover(tc, graph, scan):
    s, d, n, want = graph
    s2, d2 = s.repeat(2), d.repeat(2)
    eo = np.array([0, s.numel(), 2 * s.numel()], np.int64)
    vn = np.array([n, n], np.int32)
    tc.tc_debug_set_wait_limit(2000)
    tc.tc_debug_set_unpublished_scan(scan, 70)  # of 129: in the second graph
    try:
        expect_timeout(tc, tc.tc_count_batch, s2, d2, eo, vn)
        with tc.Engine(2 * s.numel(), 2 * n, 4) as eng:
            for _ in range(2):  # an engine that failed is still usable
                expect_timeout(tc, eng.count, s2, d2, eo, vn)
    finally:
        tc.tc_debug_reset()
    with tc.Engine(2 * s.numel(), 2 * n, 4) as eng:
        assert list(eng.count(s2, d2, eo, vn)) == [want["T"]] * 2
    assert list(tc.tc_count_batch(s2, d2, eo, vn)) == [want["T"]] * 2


def test_a_lowered_limit_alone_keeps_the_sorts_that_calls_use(tc, graph):
    """A call sorts the same way with any wait limit: as many kernels launch."""
    s, d, n, want = graph
    seen = []
    try:
        for limit in (1 << 24, 1 << 20):
            tc.tc_debug_set_wait_limit(limit)
            before = tc.tc_launch_count()
            assert tc.tc_count(s, d, n) == want["T"]
            seen.append(tc.tc_launch_count() - before)
    finally:
        tc.tc_debug_reset()
    assert seen[0] == seen[1]
