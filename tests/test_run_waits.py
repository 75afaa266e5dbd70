"""What a whole run does after a wait has given up, read from the source: a block that stands still for seconds cannot be had
on a GPU without a fault."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0912_2555_gb300", "csrc")


def test_the_grid_kernel_leaves_nothing_behind_a_wait_that_gave_up():
    """A block that gave up at the barrier after the renumbering writes no reader lists; the others give up at the next
    barrier, k_own's last.  The graph must not be left to k_tail then: it would take unwritten words as addresses."""
    with open(os.path.join(CSRC, "map_run.cuh")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    body = text[text.index(" k_own("):text.index("struct PrepareOut")]
    last = body.rindex("alive = run_barrier(")
    hand = body.index("c->hand = 2")
    assert last < hand
    condition = body[body.rindex("if (", 0, hand):hand].split("{")[0]
    assert "hand" in condition and "alive" in condition
