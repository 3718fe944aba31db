"""Blocks of a cluster may write one another's shared memory only once all of them run: in the kernel launched as a
cluster, a barrier that all blocks pass precedes the first access through map_shared_rank.  Read from the source, since
a block that starts late enough to be missed cannot be arranged in a run.
"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_11130_gb300", "csrc")


def test_every_cluster_kernel_is_known():
    found = {f for f in os.listdir(CSRC) if "__cluster_dims__" in open(os.path.join(CSRC, f)).read()}
    assert found == {"coarse_inverse.cu"}


def test_barrier_before_the_first_remote_access():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "coarse_inverse.cu")).read())
    body = src[src.index(" panel_kernel(PanelArgs g) {"):src.index("pivot_rows_kernel")]
    columns = body.index("for (int c = 0; c < g.nb")
    assert columns < body.index("map_shared_rank")
    before = body[:columns]                     # a barrier inside the loop comes too late for the first column
    assert ".sync()" in before or ".barrier_wait()" in before
