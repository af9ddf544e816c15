"""Vertices whose degree, counted with repeated pairs, has more bits than the
rank keys' digits (csrc/preprocess.cu, k_rank_keys; calls that sort by radix
passes): they still come last in the order, so no forward list exceeds sqrt(2m)
entries.  Two hubs joined to each other and to every other vertex, each pair
given so often that the hubs' degree is exactly 2^24 (of 24 bits: zero) or
more.  By hand: T = n - 2, one triangle per other vertex."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LEAVES, COPIES, JOINED = 99864, 168, 64  # 99864 * 168 + 64 = 2^24


@pytest.mark.parametrize("more", [0, 200])
def test_two_hubs_of_degree_two_to_the_24(more):
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_1503_00576_gb300 as tc

    n = LEAVES + 2
    assert LEAVES * COPIES + JOINED == 1 << 24
    leaf = torch.arange(2, n, dtype=torch.int32, device="cuda").repeat(COPIES)
    hub = torch.zeros_like(leaf)
    joined = torch.zeros(JOINED + more, dtype=torch.int32, device="cuda")
    s = torch.cat([hub, hub + 1, joined])
    d = torch.cat([leaf, leaf, joined + 1])
    assert tc.tc_count(s, d, n) == LEAVES
    T, t, deg = tc.tc_count_per_vertex(s, d, n)
    assert T == LEAVES
    want_t, want_deg = np.ones(n, np.int64), np.full(n, 2, np.int32)
    want_t[:2], want_deg[:2] = LEAVES, LEAVES + 1
    assert np.array_equal(t.cpu().numpy(), want_t)
    assert np.array_equal(deg.cpu().numpy(), want_deg)
