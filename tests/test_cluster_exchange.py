"""What the blocks of a cluster send each other in a short prefill: rules that no run shows to be broken, checked in the sources.  No GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_05431_b200", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _function(text, name):
    """The body of a function: from its name to the closing brace in the first column."""
    return re.search(r"\b" + name + r"\(.*?\n}\n", text, flags=re.S).group(0)


def test_rows_from_other_blocks_are_waited_for_at_the_scope_of_the_cluster():
    """The copies and stores of the other blocks complete on `bar_recv` with release at cluster scope; a wait without a scope of its own acquires at
    the scope of the block, behind which their bytes need not be visible."""
    common, attn = _source("ape_common.cuh"), _source("ape_attn.cu")
    assert "mbarrier.try_wait.parity.acquire.cluster." in _function(common, "mbar_try_wait_cluster")
    waits = re.findall(r"\bmbar_\w*wait\w*(<\w+>)?\(bar_recv\b", attn)
    assert waits == ["<true>"]
    assert "CLUSTER ? mbar_try_wait_cluster(bar, parity)" in _function(common, "mbar_wait")
