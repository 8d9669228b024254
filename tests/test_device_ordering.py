"""Orderings that a run cannot be relied on to show (the hardware's schedule hides them), read off
the kernel and runtime sources.  CPU."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_18491_gb300", "csrc")
BARRIER = re.compile(r"__syncwarp\(|__syncthreads\(|bar\.sync")


def _sources():
    """(name, text without comments) of every source file."""
    out = []
    for f in sorted(glob.glob(os.path.join(CSRC, "*"))):
        if f.endswith((".cu", ".cuh", ".cpp", ".h")):
            text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(f).read(), flags=re.S)
            out.append((os.path.basename(f), text))
    assert len(out) > 10
    return out


def test_shared_memory_filled_by_other_lanes_is_read_behind_a_barrier():
    """cp.async.wait_group covers the executing thread's own copies: between it and the first read of
    shared memory stands a barrier of the threads that copied; likewise between the reads of a stage
    and the copies that fill it again."""
    seen = 0
    for name, text in _sources():
        for m in re.finditer(r"cp\.async\.wait_group", text):
            rest = text[m.end():]
            read = re.search(r"ld\.shared|lds_", rest)
            if not read:
                continue
            seen += 1
            assert BARRIER.search(rest[:read.start()]), "%s: shared read behind wait_group without a barrier" % name
        # a loop that refills its stages: the barrier stands before the call
        for m in re.finditer(r"\n[^\n]*\n\s*if \(!fetch\(\)\)", text):
            seen += 1
            assert BARRIER.search(m.group(0)), "%s: a stage is refilled without a barrier" % name
    assert seen >= 2


def test_uploads_run_on_the_stream_that_reads_them():
    """A cudaMemcpy from pageable memory or a cudaMemset runs on the legacy stream and may return
    before it has landed; a non-blocking stream is not ordered behind it.  So device memory is
    written by the asynchronous forms on the reading stream, and symbols are followed by a wait."""
    for name, text in _sources():
        for m in re.finditer(r"\bcudaMemcpy\s*\(", text):
            call = text[m.start():text.index(";", m.start())]
            assert "DeviceToHost" in call, "%s: %s" % (name, call)
        assert not re.search(r"\bcudaMemset\s*\(", text), name
        last = text.rfind("cudaMemcpyToSymbol(")
        assert last < 0 or "cudaStreamSynchronize(cudaStreamLegacy)" in text[last:], name
