"""Orderings that the task kernel's shared counters rely on, read from its source:
no run on one machine shows a missing one."""
import os

import bench

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1602_02864_gb300", "csrc")


def body(text, signature):
    """The text of a function from its signature to the brace that closes it."""
    at = text.index(signature)
    depth = 0
    for i in range(text.index("{", at), len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at:i + 1]
    raise AssertionError(signature)


def kernel_source():
    with open(os.path.join(CSRC, "rows_kernel.cuh")) as f:
        return bench.code_tokens(f.read())


def in_order(text, *parts):
    at = 0
    for p in parts:
        at = text.index(p, at) + len(p)


def test_last_warp_sees_every_status_and_arrival():
    """A warp's arrival at the launch's end is a release; the last warp fences between seeing
    all arrivals and reading the status word (lane 0 sees them, so a warp barrier follows)."""
    src = kernel_source()
    assert "atom.inc.release.gpu" in body(src, "unsigned int atom_inc_release(")
    end = body(src, "void warp_done(")
    assert "atomicInc" not in end
    in_order(end, "atom_inc_release(&ga.ctl->done", "return;", "__threadfence();", "__syncwarp();", "__ldcg(ga.status)")


def test_combining_warp_reads_partials_after_their_arrivals():
    """The segments' partials are written before a release arrival, and the warp that adds them
    puts a fence and a warp barrier between lane 0's arrival and every lane's reads."""
    src = kernel_source()
    in_order(body(src, "int segment_done("), "__syncwarp();", "atom_inc_release(a.seg_done")
    in_order(src[src.index("ready >= 0"):], "__threadfence();", "__syncwarp();", "combine_row(")


def test_task_length_across_two_to_the_31(tmp_path):
    """The length of a task from the low words of its ends, where an odd multiple of 2^31
    nonzeros lies between them: evaluated as a constant, in which a signed overflow is an error."""
    import subprocess
    from paper_1602_02864_gb300 import build
    src = tmp_path / "len.cu"
    src.write_text('#include "internal.h"\n'
                   "using spmm::entries_between;\n"
                   "constexpr int top = 0x7fffff00, low = -0x7fffff00;\n"
                   'static_assert(entries_between(top, low) == 512, "across 2^31");\n'
                   'static_assert(entries_between(-256, 256) == 512, "across 2^32");\n'
                   'static_assert(entries_between(5, 5) == 0 && entries_between(5, 517) == 512, "plain");\n')
    subprocess.check_call([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-c", str(src), "-o", str(tmp_path / "len.o")])
    src = kernel_source()
    assert "n = entries_between(e0, x.end.x)" in src and "x.end.x - e0" not in src
