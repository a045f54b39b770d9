"""Prefill of the per-context form and of trees with so few nodes that one pass with a partial per node serves: node counts on both sides of
that line, ragged and empty nodes, against the oracle and against the two-pass form, which an SM budget of one selects."""
import pytest
import torch

from oracle import ape_oracle as orc
from paper_2502_05431_b200 import libape
from paper_2502_05431_b200 import workloads as wl
from tests.gpu_util import compare, gpu_attend, handle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["per_context", "tree"])
@pytest.mark.parametrize("kw", [
    dict(H_q=32, H_kv=8, d=128, l_P=20, ctx_lens=[[300, 1, 0, 129, 128, 64, 700]], l_q=33, l_k=40),          # six with tokens
    dict(H_q=32, H_kv=8, d=128, l_P=20, ctx_lens=[[300, 1, 5, 129, 128, 64, 700]], l_q=33, l_k=40),          # seven
    dict(H_q=4, H_kv=1, d=64, l_P=0, ctx_lens=[[40], [2000, 3], [77, 5, 6, 1, 1]], l_q=70, l_k=70, gap=3),
    dict(H_q=8, H_kv=2, d=128, l_P=130, ctx_lens=[[129, 400], [1, 1]], l_q=300, l_k=301),                    # siblings
])
def test_few_nodes(form, kw):
    b = wl.make_batch(seed=51, T=0.8, S=0.6, name=form, **kw)
    parents = [[-1 if i % 3 == 0 else i - i % 3 for i in range(len(rq.ctx))] for rq in b.requests]
    how = dict(per_context=True) if form == "per_context" else dict(tree=(parents, None))
    out, lse, n = gpu_attend(b, libape.APE_PREFILL, **how)
    assert n == (4 if 5 in kw["ctx_lens"][0] else 2)           # (seven with tokens: two passes)
    handle().set_sm_budget(1)
    try:
        two, two_lse, n = gpu_attend(b, libape.APE_PREFILL, **how)
    finally:
        handle().set_sm_budget(0)
    assert n == 4
    compare(out, two.float(), "one pass against two")
    assert (lse - two_lse).abs().max() < 1e-3
    for r, rq in enumerate(b.requests):
        q, p, c, k = b.views(r)
        ref = orc.attend(q, p, c, k, b.T, b.S, per_context=True) if form == "per_context" else orc.attend_tree(q, p, c, k, b.T, b.S, parents[r], None)
        sl = slice(rq.q_start, rq.q_start + rq.q_len)
        compare(out[sl], ref.out.float(), f"{form} req {r}")
        assert (lse[sl].double() - ref.lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("H_q,H_kv,d,n_req,nodes,l_q,kernels", [
    (32, 8, 128, 1, [256] * 3, 64, 2), (32, 8, 128, 1, [256] * 5, 64, 4),          # 4.2 against 5.4, 7.0 against 5.4
    (32, 8, 128, 1, [512] * 5, 128, 4), (32, 8, 128, 1, [1100] * 5, 128, 2),       # two waves of rows: 10.2 against 7.4 and 12.4
    (32, 8, 128, 2, [31] * 3, 37, 2), (32, 8, 128, 2, [31] * 3, 38, 4),            # 4.35 and 4.41 against 4.4
    (8, 8, 128, 1, [40] * 4, 3, 2),
    (8, 2, 64, 1, [256] * 6, 64, 2), (8, 2, 64, 1, [100] * 6, 64, 2), (8, 2, 64, 1, [100] * 6, 400, 4),
])
def test_trees_whose_walk_is_worth_it(H_q, H_kv, d, n_req, nodes, l_q, kernels):
    """Where the walk over a tree's nodes costs more than the two kernels and the pass that it saves (148 SMs), the plan keeps them."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the rows of a wave are those of 148 SMs")
    b = wl.make_batch(H_q=H_q, H_kv=H_kv, d=d, l_P=20, ctx_lens=[nodes] * n_req, l_q=l_q, seed=52, T=0.8, S=0.6, name="walk")
    parents = [[-1] + [0] * (len(nodes) - 1)] * n_req
    dev = b.to("cuda:0")
    plan = handle().attend_plan(H_q=H_q, H_kv=H_kv, d=d, k_pool=dev.k_pool, v_pool=dev.v_pool, q=dev.q, out=torch.zeros_like(dev.q),
                                requests=b.requests, mode=libape.APE_PREFILL, tree=(parents, None))
    plan.attend(b.T, b.S, plan.alloc_workspace())
    torch.cuda.synchronize()
    assert plan.last_kernels() == kernels
    out, lse, _ = gpu_attend(b, libape.APE_PREFILL, tree=(parents, None))
    for r, rq in enumerate(b.requests):
        ref = orc.attend_tree(*b.views(r), b.T, b.S, parents[r], None)
        sl = slice(rq.q_start, rq.q_start + rq.q_len)
        compare(out[sl], ref.out.float(), f"req {r}")
        assert (lse[sl].double() - ref.lse).abs().max().item() < 2e-3
