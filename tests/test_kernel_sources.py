"""Rules that the kernels' sources keep, on the CPU.

Runs of few pairs launch every kernel early: its blocks are resident while the
kernels before it still write what it is going to read, and wait in
grid_begin().  Read-only loads (ld.global.nc, __ldg, const __restrict__) are for
data that no one writes during the life of a kernel, so no kernel may use them,
and every kernel has to wait before anything else."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1503_00576_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def code(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_read_only_loads(path):
    text = code(path)
    assert not re.search(r"ld\.global[.\w:]*\.nc\b", text)
    assert "__ldg" not in text
    assert not re.search(r"const\s+[\w\s]*\*\s*__restrict__", text)


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_every_kernel_waits_first(path):
    text = code(path)
    kernels = re.findall(r"__global__[^{;]*?\b(k_\w+)\s*\([^{;]*\)\s*\{\s*([^\n]*)", text)
    assert len(kernels) == len(re.findall(r"__global__", text))
    for name, first in kernels:
        assert first.strip() == "grid_begin();", name


def test_hub_product_leaves_its_tile_loop_by_a_vote():
    """S.abort is set by the thread that loads and the one that multiplies, in
    the next tile as soon as they have passed a tile's last barrier: a thread
    that tested it behind that barrier could leave a block that goes on."""
    text = code(os.path.join(CSRC, "hub.cu"))
    body = text[text.index("k_hub_gemm("):text.index("k_hub_finish(")]
    loop = body[body.index("for (uint32_t tile"):body.index("tcgen05.dealloc")]
    reads = re.findall(r"[^\n]*S\.abort(?!\s*=)[^\n]*", loop)
    assert [r.strip() for r in reads] == [
        "const bool ok = mbar_wait(&S.done, parity) && !S.abort;",  # before the tile's barriers
        "if (__syncthreads_or(!ok || S.abort)) {"]
