"""Merge of the partials: rows whose partials are shared by eight warps and rows with one, and rows with more partials than one round of
lanes covers.  The number of partials per row follows the SM budget (one KV head: every thread block leaves one or two)."""
import pytest
import torch

from paper_2502_05431_b200 import libape
from paper_2502_05431_b200 import workloads as wl
from tests.gpu_util import compare, gpu_attend, handle, oracle_attend

pytestmark = pytest.mark.gpu


def _check(b, mode, **kw):
    out, lse, n = gpu_attend(b, mode, **kw)
    for r, rq in enumerate(b.requests):
        ref = oracle_attend(b, r)
        sl = slice(rq.q_start, rq.q_start + rq.q_len)
        compare(out[sl], ref.out.float(), f"{b.name} req {r}")
        assert (lse[sl].double() - ref.lse).abs().max().item() < 2e-3
    return n


@pytest.mark.parametrize("n_sm", [1, 6, 7, 8, 14, 15, 16, 33, 0])
@pytest.mark.parametrize("mode,d,l_q", [(libape.APE_DECODE, 128, 1), (libape.APE_PREFILL, 64, 19), (libape.APE_PREFILL, 128, 150)])
def test_partials_per_row(n_sm, mode, d, l_q):
    """(4 rows, 256 slot rows: eight warps a row; 768 slot rows: one)"""
    b = wl.make_batch(H_q=4, H_kv=1, d=d, l_P=70, ctx_lens=[[3000, 1, 2999]], l_q=l_q, l_k=l_q + 40, seed=31, T=0.8, S=0.9,
                      name=f"merge_sm{n_sm}")
    handle().set_sm_budget(n_sm)
    try:
        _check(b, mode)
    finally:
        handle().set_sm_budget(0)


@pytest.mark.parametrize("n_sm", [3, 24, 60, 100, 146])
@pytest.mark.parametrize("d,H_q,H_kv,n_req,l_q", [(64, 8, 8, 3, 3), (128, 32, 8, 3, 20), (128, 16, 4, 5, 9), (64, 32, 2, 10, 17)])
def test_more_rows_than_warps(n_sm, d, H_q, H_kv, n_req, l_q):
    """5,120 or 6,144 slot rows, more than there are places for a warp per row: eight lanes share a row, up to eight partials a segment."""
    b = wl.make_batch(H_q=H_q, H_kv=H_kv, d=d, l_P=70, ctx_lens=[[900 - 100 * r] for r in range(n_req)] if n_req < 9 else [[500]] * n_req, l_q=l_q,
                      l_k=l_q + 40, seed=34, T=0.8, S=0.9, name=f"merge_rows_sm{n_sm}")
    handle().set_sm_budget(n_sm)
    try:
        _check(b, libape.APE_PREFILL)
    finally:
        handle().set_sm_budget(0)


def test_more_partials_than_one_round_of_lanes():
    """One KV head and a shared-context batch of at most 128 rows, two tiles per thread block: two partials per block, 296 per row on
    148 SMs, of which the eight warps of a row take 256 in one round."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    b = wl.share_contexts(wl.make_batch(H_q=4, H_kv=1, d=128, l_P=5, ctx_lens=[[2 * n_sm * 128]] + [[1]] * 5, l_q=1, l_k=9, seed=32,
                                        T=0.9, S=0.8, name="merge_296"))
    dev = b.to("cuda:0")
    plan = handle().attend_plan(H_q=4, H_kv=1, d=128, k_pool=dev.k_pool, v_pool=dev.v_pool, q=dev.q, out=torch.zeros_like(dev.q),
                                requests=b.requests, mode=libape.APE_DECODE, shared=True)
    # a slot holds two partials of 128 rows; what the requests' own segments add is less than three slots
    assert 2 * (plan.workspace_bytes // (256 * (128 + 2) * 4) - 3) > 256
    assert _check(b, libape.APE_DECODE, shared=True) == 3              # rest, context pass, merge


@pytest.mark.parametrize("n_sm", [16, 15, 17, 40, 147])
def test_runs_with_thread_blocks_of_their_own(n_sm):
    """Eight heads, a long and a short segment each: budgets at which every (head, segment) gets its own thread blocks (16: one
    each), the one below at which that does not fit, and budgets with tiles to spare."""
    b = wl.make_batch(H_q=8, H_kv=8, d=128, l_P=70, ctx_lens=[[60, 1, 130, 64]], l_q=1, l_k=9, gap=3, seed=33, T=0.8, S=0.9,
                      name=f"own_blocks_sm{n_sm}")
    handle().set_sm_budget(min(n_sm, torch.cuda.get_device_properties(0).multi_processor_count - 1))
    try:
        assert _check(b, libape.APE_DECODE) == 2                        # (no clusters under a budget)
    finally:
        handle().set_sm_budget(0)
