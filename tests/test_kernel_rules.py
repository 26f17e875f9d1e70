"""Rules that the kernels' sources keep where a run cannot show a breach: an
ordering or a wait that is missing goes right as long as the hardware happens
to order things so."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_20532_gb300", "csrc")


def _source(name):
    """A source file without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _function(text, name):
    """The body of the function `name`, by its braces."""
    at = re.search(r"\b%s\([^;{]*\)\s*\{" % name, text)
    assert at, name
    depth, i = 1, at.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[at.end():i - 1]


def test_tensor_memory_follows_a_warp_wide_wait():
    """Tensor memory is written and read after a bounded wait that the whole
    warp leaves together and that a tcgen05 fence follows."""
    text = _source("verify_tc.cu")
    wait = _function(text, "tc_wait")
    order = [wait.find(k) for k in ("mbar_wait_bounded", "tcgen05.fence::after_thread_sync", "return")]
    assert "__all_sync(FULL, mbar_wait_bounded(" in wait
    assert -1 not in order and order == sorted(order)
    assert text.count("mbar_wait_bounded(") == 1, "every wait of the kernel goes through tc_wait"
    kernel = _function(text, "verify_tc_kernel")
    for use in ("tc_store32(", "tc_load32("):
        assert 0 <= kernel.find("tc_wait(") < kernel.find(use)


def test_early_kernels_load_coherently():
    """A kernel that begins with pdl_wait() may be set up while kernels before
    it still write what it reads, so neither it nor the device code it shares
    uses the read-only path."""
    files = [f for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))]
    early = [f for f in files if re.search(r"\bpdl_wait\(", _source(f)) or f in ("elim.cuh", "full.cuh")]
    assert {"learn.cu", "store.cu", "merge.cu", "host_io.cu", "verify_tc.cu", "elim_wide.cu"} <= set(early)
    for f in early:
        text = _source(f)
        assert not re.search(r"__ldg\(|ld\.global\.nc", text), f
        for kernel in re.finditer(r"__global__[^{;]*?\w+\(([^{;]*)\)\s*\{", text):
            assert "__restrict__" not in kernel.group(1), (f, kernel.group(1))
