"""mpcd_collide_solvent_static returns before its kernel has run, so a wait inside the kernel
that gave up could not be told to the caller, who would go on with a collision done in
part: its barriers are those of the cluster and of the cooperative grid, which do not
give up (all their CTAs are resident, or the launch is refused)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_14307_gb300", "csrc")


def function(text, name):
    """The body of the function `name`, braces matched."""
    at = text.index("{", re.search(r"\b%s\(" % name, text).start())
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == "{") - (text[i] == "}")
        if depth == 0:
            return text[at:i + 1]


def test_no_wait_that_gives_up():
    src = open(os.path.join(CSRC, "kernels_solvent.cu")).read()
    barrier, kernel = function(src, "box_barrier"), function(src, "k_collide_box")
    assert "this_grid().sync()" in barrier and "barrier.cluster.wait" in barrier
    for text in (barrier, kernel, open(os.path.join(CSRC, "static_collide.cu")).read()):
        for word in ("SPIN_LIMIT", "ERR_TIMEOUT", "ld.acquire", "d_err", "while (seen"):
            assert word not in text, word
    assert kernel.count("box_barrier<CLUSTER>();") == 2 and "return;" not in kernel
