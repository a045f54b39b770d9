"""What the blocks of a cluster send each other in a short prefill: rules that no run shows to be broken, checked in the sources and by a model
of two blocks.  No GPU."""
import os
import re
import subprocess

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
    waits = re.findall(r"\b(mbar_\w*wait\w*)\(bar_recv\b", attn)
    assert waits == ["mbar_wait_received"]
    assert "mbar_try_wait_cluster(bar, 0)" in _function(common, "mbar_wait_received")


_TWO_BLOCKS = r"""
#include <cstdio>
#include <initializer_list>
#include "ape_wait.h"
// One wait of block 0 has run out (its abort flag is up) when it comes to the rows that block 1 sends; block 1's own wait runs out later, it lets its
// copies and products drain and sends.  The clock moves with every look at it.
int main() {
    for (long long sent : {0ll, 5000ll, ape::kWaitCycles - 1, ape::kWaitCycles + 3 * (1ll << 24), 2 * ape::kWaitCycles, -1ll}) {
        long long clock = 0;
        const long long landed = sent + 4000, step = 1ll << 20;
        bool gave_up = false;
        const bool here = ape::wait_received([&] { return sent >= 0 && clock >= landed; }, [&] { return clock += step; }, [&] { gave_up = true; });
        if (sent >= 0 && (!here || gave_up || clock < landed)) return std::printf("left at %lld, rows land at %lld\n", clock, landed), 1;
        if (sent < 0 && (here || !gave_up || clock > ape::kReceiveCycles + 2 * step)) return std::printf("no limit\n"), 2;
    }
    return 0;
}
"""


def test_no_block_leaves_before_what_is_sent_to_it_has_landed(tmp_path):
    """A block whose waits have run out is sent its rows, too, perhaps by blocks that come to it later: it waits for them longer than any of their own
    waits can last, but not for ever.  And its sends depend on nothing that an abort changes: the others count on them."""
    src = tmp_path / "two_blocks.cpp"
    src.write_text(_TWO_BLOCKS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(tmp_path / "two_blocks")], check=True)
    r = subprocess.run([str(tmp_path / "two_blocks")], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
    attn = _source("ape_attn.cu")
    body = _function(_source("ape_common.cuh"), "mbar_wait_received")
    assert "wait_received(" in body and "if" not in body
    exchange = attn[attn.index("cluster_send2("):attn.index("mbar_wait_received(bar_recv")]
    assert "ok" not in re.findall(r"\w+", exchange) and "abort_flag" not in exchange
    # the wait comes before the block's arrival at the last barrier of the cluster
    assert attn.index("mbar_wait_received(bar_recv") < attn.index("cluster_arrive_relaxed();", attn.index("cluster_send2("))
