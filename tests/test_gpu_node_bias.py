"""The walk between the two passes of a prefill over context trees: levels of very different widths, children whose breadth-first
order differs from their index order, the deepest tree, and as many nodes as the shared-memory form of the walk takes."""
import random
import threading

import pytest
import torch

from paper_2502_05431_b200 import libape
from paper_2502_05431_b200 import workloads as wl
from tests.gpu_util import handle
from tests.test_gpu_tree import _check

pytestmark = pytest.mark.gpu
HEADS = dict(H_q=4, H_kv=2, d=64)


def _interleaved(n, n_roots):
    """Node i >= n_roots is a child of node i mod n_roots, or of that child's first child."""
    return [-1 if i < n_roots else (i % n_roots if i < 2 * n_roots else n_roots + i % n_roots) for i in range(n)]


def _run(lens, parents, scaled, l_q=17):
    b = wl.make_batch(**HEADS, l_P=9, ctx_lens=lens, l_q=l_q, seed=80, T=0.8, S=0.7, name="node_bias")
    _check(b, libape.APE_PREFILL, parents, scaled)


def test_interleaved_children_and_marks_at_every_level():
    rnd = random.Random(5)
    lens = [[rnd.choice([0, 1, 5, 40]) for _ in range(90)]]
    lens[0][-1] = 7
    _run(lens, [_interleaved(90, 7)], [[rnd.random() < 0.5 for _ in range(90)]])


def test_deepest_tree_and_a_request_without_contexts():
    chain = list(range(-1, 15))                                     # 16 levels
    _run([[3] * 16, [], [20, 0, 4]], [chain, [], [-1, -1, 0]], None, l_q=40)


@pytest.mark.parametrize("n,parents", [(1600, [-1] * 1600), (1600, _interleaved(1600, 3)), (1701, [-1] * 1701), (1750, _interleaved(1750, 40))])
def test_as_many_nodes_as_fit_and_more(n, parents):
    """(1,709 nodes x 136 bytes is what a block's shared memory holds)"""
    _run([[1 + i % 3 for i in range(n)]], [parents], None, l_q=3)


def test_two_threads_with_trees_of_different_sizes():
    """The walk's launch asks for shared memory by the number of nodes: one thread's small tree must not lower the limit between the two
    steps (limit, launch) of another thread's large one."""
    errors = []

    def work(n):
        try:
            torch.cuda.set_device(0)
            b = wl.make_batch(**HEADS, l_P=9, ctx_lens=[[1] * n], l_q=1, seed=81, T=0.8, S=0.7, name="threads").to("cuda:0")
            out = torch.zeros_like(b.q)
            with torch.cuda.stream(torch.cuda.Stream()):
                plan = handle().attend_plan(**HEADS, k_pool=b.k_pool, v_pool=b.v_pool, q=b.q, out=out, requests=b.requests,
                                            mode=libape.APE_PREFILL, tree=([[-1] * n], None))
                ws = plan.alloc_workspace()
                plan.attend(b.T, b.S, ws)
                torch.cuda.current_stream().synchronize()
                first = out.clone()
                for i in range(4000):
                    plan.attend(b.T, b.S, ws)
                torch.cuda.current_stream().synchronize()
                assert torch.equal(out, first)
        except Exception as e:                                        # noqa: BLE001
            errors.append(f"{n} nodes: {e!r}")

    threads = [threading.Thread(target=work, args=(n,)) for n in (1600, 400)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not errors, errors
