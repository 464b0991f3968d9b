"""The batch rebuilds its work lists whenever a domain leaves or rejoins it.  They are
allocated once, at the start, for the longest that any active set can have: an allocation that
fails in between would leave the step with a list that is not there."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1405_2232_gb300", "csrc")


def test_rebuilding_the_lists_allocates_nothing():
    s = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "lb_batch.cu")).read())
    body = s[s.index("lb_status rebuild_lists("):s.index("void release(lb_batch* b)")]
    assert "cudaMemcpyAsync" in body and not re.search(r"cuda(Malloc|Free)", body)
