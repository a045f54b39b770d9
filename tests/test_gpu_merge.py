"""Merge of the partials: rows whose partials are shared by eight warps and rows with one, and rows with more partials than one round of
lanes covers.  The number of partials per row follows the SM budget (one KV head: every thread block leaves one or two)."""
import pytest
import torch

from oracle import ape_oracle as orc
from paper_2502_05431_b200 import libape
from paper_2502_05431_b200 import workloads as wl
from tests.gpu_util import compare, gpu_attend, handle, kernels_in_order, oracle_attend
from tests.test_gpu_sharded import _sharded as sharded

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
    """5,120 to 10,240 slot rows, more than there are places for a warp per row: eight lanes share a row, of up to four partials a segment."""
    b = wl.make_batch(H_q=H_q, H_kv=H_kv, d=d, l_P=70, ctx_lens=[[900 - 100 * r] for r in range(n_req)] if n_req < 9 else [[500]] * n_req, l_q=l_q,
                      l_k=l_q + 40, seed=34, T=0.8, S=0.9, name=f"merge_rows_sm{n_sm}")
    handle().set_sm_budget(n_sm)
    try:
        _check(b, libape.APE_PREFILL)
    finally:
        handle().set_sm_budget(0)


def _merge_and_partials(b, **how):
    """The last kernel of a prefill, and how many partials of its context segment a row has on average (a partial more is the rest's)."""
    dev = b.to("cuda:0")
    plan = handle().attend_plan(H_q=b.H_q, H_kv=b.H_kv, d=b.d, k_pool=dev.k_pool, v_pool=dev.v_pool, q=dev.q, out=torch.zeros_like(dev.q),
                                requests=b.requests, mode=libape.APE_PREFILL, **how)
    ws = plan.alloc_workspace()
    slots = plan.workspace_bytes // (256 * (b.d + 2) * 4)
    kernels = kernels_in_order(lambda: plan.attend(b.T, b.S, ws))
    plan.close()
    return kernels, slots / (len(b.requests) * b.H_kv) - 1


@pytest.fixture
def budget():
    """Plans for so many of 148 SMs, so that a context segment is cut into a known number of partials."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the line between the merge kernels is that of 148 SMs")
    yield handle().set_sm_budget
    handle().set_sm_budget(0)


def _nineteen_heads(d, lens, **kw):
    """19 KV heads of three query rows: 4,864 slot rows to merge, the fewest above the line of 4,736; one tile beside the contexts."""
    return wl.make_batch(H_q=76, H_kv=19, d=d, l_P=0, ctx_lens=lens, l_q=3, l_k=3, seed=35, T=0.8, S=0.9, name="nineteen", **kw)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n_sm,tiles,most,kernel", [(84, 80, 5, "merge_rows"), (139, 80, 6, "merge_rows"), (128, 80, 7, "merge_rows"),
                                                    (147, 80, 8, "merge_rows"), (147, 200, 9, "merge")])
def test_rows_of_five_to_nine_partials(budget, d, n_sm, tiles, most, kernel):
    """Eight lanes to a row read its partials three at a time, eight at most: two and three batches, the last one full or not; with nine a warp takes the
    row.  Eight lanes are only taken for at most eight, so the kernel and the average together say how many there are."""
    b = _nineteen_heads(d, [[128 * tiles]])
    budget(n_sm)
    kernels, partials = _merge_and_partials(b)
    assert kernels == ["attn", kernel] and most - 1 < partials <= most
    _check(b, libape.APE_PREFILL)


@pytest.mark.parametrize("d", [64, 128])
def test_empty_partials_of_rows_that_eight_lanes_merge(budget, d):
    """A partial whose sum of weights is no positive number is empty: all partials of a head with NaN in its query (zeros, minus infinity), one of eight
    where a key is NaN (the rest of the mass is there), and nothing else changes."""
    b = _nineteen_heads(d, [[128 * 80]])
    b.T = b.S = 1.0
    budget(147)
    assert _merge_and_partials(b)[0] == ["attn", "merge_rows"]
    clean, clean_lse, _ = gpu_attend(b, libape.APE_PREFILL)
    b.q[1, 7] = float("nan")
    out, lse, _ = gpu_attend(b, libape.APE_PREFILL)
    assert (out[1, 7] == 0).all() and lse[1, 7] == float("-inf")
    out[1, 7], lse[1, 7] = clean[1, 7], clean_lse[1, 7]
    assert torch.equal(out, clean) and torch.equal(lse, clean_lse)
    b = _nineteen_heads(d, [[128 * 80]])
    b.T = b.S = 1.0
    for tok in (0, 5000, 128 * 80 - 1):                          # in the first, one of the middle, the last partial of KV head 3
        kv = wl.Batch(b.H_q, b.H_kv, b.d, b.q, b.k_pool.clone(), b.v_pool, b.requests, b.T, b.S, None, b.name, {})
        kv.k_pool[b.requests[0].ctx[0][0] + tok, 3] = float("nan")
        out, lse, _ = gpu_attend(kv, libape.APE_PREFILL)
        assert torch.isfinite(out.float()).all()
        left = (lse[:, 12:16] - clean_lse[:, 12:16]).exp()        # of the weights of a row, without the partial's 7 to 13 of 81 tiles
        assert (left > 0.5).all() and (left < 0.99).all()
        out[:, 12:16], lse[:, 12:16] = clean[:, 12:16], clean_lse[:, 12:16]
        assert torch.equal(out, clean) and torch.equal(lse, clean_lse)


def test_no_context_and_row_blocks_that_see_nothing(budget):
    """No context segment; and the causal query segment of 18 row blocks is cut where its first row blocks see none of what is behind the cut: their
    partials there are empty and their rows were never written."""
    b = wl.make_batch(H_q=32, H_kv=8, d=128, l_P=0, ctx_lens=[[]], l_q=1100, l_k=1100, seed=36, T=0.8, S=0.9, name="causal")
    budget(147)
    assert _merge_and_partials(b)[0] == ["attn", "merge_rows"]
    _check(b, libape.APE_PREFILL)


def test_two_passes_that_end_with_eight_lanes_to_a_row(budget):
    b = wl.make_batch(H_q=16, H_kv=4, d=128, l_P=0, ctx_lens=[[640] * 8] * 5, l_q=3, l_k=3, seed=37, T=0.8, S=0.6, name="two_pass")
    budget(147)
    kernels, _ = _merge_and_partials(b, per_context=True)
    assert kernels[-1] == "merge_rows" and len(kernels) == 4
    out, lse, _ = gpu_attend(b, libape.APE_PREFILL, per_context=True)
    for r, rq in enumerate(b.requests):
        ref = orc.attend(*b.views(r), b.T, b.S, per_context=True)
        sl = slice(rq.q_start, rq.q_start + rq.q_len)
        compare(out[sl], ref.out.float(), f"two passes req {r}")
        assert (lse[sl].double() - ref.lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("d", [64, 128])
def test_shards_whose_segments_eight_lanes_merge(budget, d):
    """A shard of a context-sharded attend hands out the two segments of a row instead of the merged one."""
    b = _nineteen_heads(d, [[2000, 3120]], gap=1)
    budget(120)
    assert _merge_and_partials(b)[0] == ["attn", "merge_rows"]       # (the form of a shard's plan, too: fewer tiles, the same rows)
    out, lse = sharded(b, libape.APE_PREFILL, 2)
    ref = oracle_attend(b, 0)
    compare(out, ref.out.float(), "shards")
    assert (lse.double() - ref.lse).abs().max().item() < 2e-3


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
