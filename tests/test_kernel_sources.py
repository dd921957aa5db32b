"""Rules of the kernel sources that no run can show safely: breaking them hangs or corrupts instead of failing."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_09936_b200", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def kernels(name):
    """(kernel name, body without comments) of every __global__ function of a source file."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)
    for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^)]*\)\s*)?(\w+)\(", text):
        start = text.index("{", m.end())
        depth, i = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
            if depth == 0:
                break
        yield m.group(1), text[start:i]


def test_every_kernel_is_found():
    found = {k for name in SOURCES for k, _ in kernels(name)}
    assert {"decode_kernel", "host_moves_kernel", "prefill_scores_kernel", "nominate_kernel", "steady_compress_kernel",
            "select_kernel", "append_kernel"} <= found


@pytest.mark.parametrize("name", SOURCES)
def test_tensor_memory_is_allocated_behind_the_wait_for_the_preceding_kernel(name):
    """A kernel that allocates first may hold, on a shared SM, the columns its own predecessor still has to get: both wait
    for ever, and no bounded wait covers an allocation."""
    for kernel, body in kernels(name):
        at = body.find("tmem_alloc(")
        if at >= 0:
            assert 0 <= body.find("pdl_wait()") < at, kernel


@pytest.mark.parametrize("name", SOURCES)
def test_products_and_their_commits_are_issued_by_the_elected_thread(name):
    """A commit covers the products of the thread that issues it.  Another thread's would report products as finished that
    still read shared memory and write tensor memory."""
    for kernel, body in kernels(name):
        guards = []   # what stands in front of the open blocks
        last = 0      # where the current statement starts
        for m in re.finditer(r"[;{}]|\b(?:umma_commit|umma_bf16)\(", body):
            if m.group() == "{":
                guards.append(body[last:m.start()])
            elif m.group() == "}":
                guards.pop()
            elif m.group() != ";":
                assert any("elect_one()" in g for g in guards + [body[last:m.start()]]), (kernel, body[last:m.end()])
                continue
            last = m.end()


def without_blocks_that_return(text):
    """What a thread that gets to the end of the text has run through."""
    while (at := text.find("return;")) >= 0:
        depth, i = 0, at
        while i >= 0 and not (text[i] == "{" and depth == 0):
            depth += {"}": 1, "{": -1}.get(text[i], 0)
            i -= 1
        depth, j = 0, at
        while j < len(text) and not (text[j] == "}" and depth == 0):
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        text = text[:i] + text[j + 1:] if i > 0 else text[:at] + text[at + len("return;"):]
    return text


@pytest.mark.parametrize("name", SOURCES)
def test_other_ctas_shared_memory_is_written_behind_a_cluster_barrier(name):
    """A CTA may write to its neighbours' shared memory, or arrive at their barriers, when all of the cluster have started: the
    whole barrier, or its waiting half, stands in front, and every thread of the CTA has arrived before its ways part."""
    for kernel, body in kernels(name):
        remote = re.search(r"\b(?:st_shared_cluster_\w+|mbar_arrive_cluster)\(", body)
        if remote:
            front = body[:remote.start()]
            run = without_blocks_that_return(front)
            assert "cluster_wait()" in run or "cluster_sync_all()" in run, kernel
            arrival = re.search(r"cluster_arrive\w*\(\)|cluster_sync_all\(\)", front).start()
            assert "return;" not in front[:arrival], kernel
