"""Kernels launched programmatically start while the kernel before them runs;
what earlier kernels wrote is visible to them only after griddepcontrol.wait.
The selection's source is read for the order of the two."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_31598_gb300", "csrc")


def kernel_body(file, name):
    """The kernel's source from its name to the next line that is a closing brace, without comments."""
    src = open(os.path.join(CSRC, file)).read()
    body = src[src.index(name + "("):]
    return re.sub(r"//[^\n]*", "", body[: body.index("\n}\n")])


def test_the_selection_and_its_append_wait_before_they_read():
    body = kernel_body("select_kernel.cu", "state_select_gather")
    wait = "ptx::pdl_wait();"
    branch, rest = body.split("return;", 1)  # the append CTAs' branch ends in the first return
    for part, reads in ((branch, ("p.frames[", "append_share<")),
                        (rest, ("p.counts[", "p.frames[", "p.positions", "p.partials"))):
        for r in reads:
            assert r in part, r
            assert wait in part[: part.index(r)], f"{r} before the wait"


def test_the_side_stream_is_joined_before_a_failed_launch_returns():
    """Recency window: once the append is on the side stream, nothing returns before the
    call's stream waits for it (no launch fails on demand, so the source is read)."""
    body = kernel_body("statekv_api.cu", "statekv_status run_step")
    forked = body[body.index("cudaEventRecord(h->ev_join"):]
    between = forked[forked.index("return STATEKV_ERR_CUDA;") + 1: forked.index("cudaStreamWaitEvent(st, h->ev_join")]
    assert "launch_attn(" in between and "return STATEKV_ERR" not in between
