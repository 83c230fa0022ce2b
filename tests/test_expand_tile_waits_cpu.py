"""Expired waits in the expand kernel of the LoRA term, from its source: on a GPU the wait in question cannot be made to run out
without leaving copies and products of other kernels in flight."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_13053_b200", "csrc")


def _without_comments(text):
    return re.sub(r"//[^\n]*", "", text)


def test_every_builder_thread_reaches_the_barriers_of_every_round():
    """The 64 threads of a group wait for an operand one by one and then meet at two barriers without a limit: a thread whose
    wait ran out may not leave the loop between them, and the tile may not pass for a result."""
    source = open(os.path.join(CSRC, "expand_tile.cuh")).read()
    loop = _without_comments(source[source.index("for (int i = group; i < nb"):source.index("where = 2;")])
    assert loop.count("bar.sync") == 2
    assert not re.search(r"\b(break|return|goto|continue)\b", loop)
    wait = loop.index("mbar_wait")
    assert wait < loop.index("*s_late = 1") < loop.index("bar.sync") < loop.index("mbarrier.arrive")
    epilogue = _without_comments(source[source.index("where = 2;"):source.index("where = 3;")])
    assert "*s_late == 0" in epilogue and not re.search(r"\b(break|return|goto|continue)\b", epilogue)
