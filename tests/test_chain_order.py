"""Orders within the kernels that no run can show to be missing, read from the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_30950_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_tensor_memory_is_taken_between_wait_and_release():
    """A chained launch that held tensor memory while it waits could starve the kernel it waits for, and
    one that let its dependents start before it holds its own could be starved by them."""
    src = source("qs_wb_row.cuh")
    body = src[src.index("wb_row_kernel(const WbParams wp)"):]
    at = [body.index(s) for s in ("chain_enter();", "chunk_setup(cb)", "chain_release();", "wb_issue_meta<DK, DV>(sm.st[0]")]
    assert at == sorted(at)
    assert body.count("chain_") == 2 and "chain_wait" not in src


def test_tensor_memory_written_by_other_threads_is_read_behind_a_fence():
    """Chunked form: u is stored to tensor memory by four warps and read by all sixteen behind a barrier;
    every reader needs the fence after it (not only the thread that issues the product)."""
    src = source("qs_chunk.cuh")
    at = src.index("tmem_st16(tl + G::kULo, ul)")
    stored = src[at:src.index("tmem_ld2x16(tl + G::kUHi, tl + G::kULo, u, ul)", at)]
    assert re.search(r"wait_st\(\);\s*\}\s*tc::fence_before_sync\(\);\s*__syncthreads\(\);\s*tc::fence_after_sync\(\);", stored)
