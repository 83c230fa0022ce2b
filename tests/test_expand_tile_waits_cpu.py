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


def _calls(file, name):
    """The argument lists of the calls of `name` in a source file."""
    source = _without_comments(open(os.path.join(CSRC, file)).read())
    return [[a.strip() for a in m.group(1).split(",")] for m in re.finditer(r"(?:return|=) " + name + r"\(([^;]*)\)[;)]", source)]


def test_both_launches_of_the_lora_term_report_to_the_workspace():
    """The status word of meteora_lora_delta's workspace takes the expired waits of its shrink and of its expand; a flag that an earlier
    call left there stays until it is read."""
    for name in ("launch_shrink", "launch_expand"):
        calls = _calls("api.cu", name)
        assert len(calls) == 1 and "ws.status" in calls[0]
    shrink = _calls("lora.cu", "launch_token_shrink")
    assert len(shrink) == 1 and shrink[0][5:8] == ["status", "false", "false"]   # (neither beside another shrink nor one of a pair)
    source = _without_comments(open(os.path.join(CSRC, "wgemm_tcgen05.cu")).read())
    assert "p.clear_status = status && pair && !beside ? 1 : 0;" in source
