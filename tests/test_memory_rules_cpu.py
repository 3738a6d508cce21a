"""Rules that memory kept between contexts rests on, held against the source: a
failed wait cannot be provoked without a fault on the device, so the calls are read.
"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = os.path.join(ROOT, "paper_1108_5673_gb300", "csrc", "pwa_abi.cu")


def code():
    text = re.sub(r"/\*.*?\*/", "", open(SOURCE).read(), flags=re.S)
    return [re.sub(r'"(\\.|[^"\\])*"|//.*', "", line) for line in text.split("\n")]


def test_buffers_of_a_call_go_back_after_a_wait_that_counts():
    """Staging, scratch and output buffers of one call: settle() directly before they are
    returned, so that a block whose last user was not waited for is never kept."""
    lines = code()
    found = 0
    for i, line in enumerate(lines):
        if re.search(r"\bdev_free\((staging|scratch|d)\)", line):
            found += 1
            assert any("settle(c)" in s for s in lines[max(0, i - 3):i]), i + 1
    assert found >= 8


def test_buffers_of_a_context_go_back_after_a_wait():
    """The first return in every function that returns a context's buffers follows quiet()."""
    lines = code()
    for i, line in enumerate(lines):
        if re.search(r"\b(dev_free|host_free)\(c->", line):
            k = i
            while re.search(r"\b(dev_free|host_free)\(c->|fx_bytes = 0|dev_alloc|return|h_fx = nullptr|pool_host_alloc|"
                            r"cudaGetLastError|^\s*[{}]*\s*$|if \(rc\)|int rc|fail\(|free_sample\(c\)|free_res\(c\)|"
                            r"cudaGraphExecDestroy|graphs", lines[k]):
                k -= 1
            assert "quiet(c)" in lines[k], (i + 1, lines[k])


def test_all_memory_is_the_pools():
    """An allocation that fails frees everything kept and is tried again: only where it is
    made through the pool, so all of them are, the model batch's plan and buffers too."""
    for i, line in enumerate(code()):
        assert not re.search(r"\b(cudaMalloc|cudaMallocHost|cudaHostAlloc|cudaFree|cudaFreeHost|cudaMallocAsync)\(",
                             line), (i + 1, line)
