"""Decode steps small enough that the blocks of a thread-block cluster merge their partials themselves: sizes at the edges of that form
(one tile, one block per segment, no context, every head layout, growth into the reserved tail), against the oracle and against the
ordinary form, which an SM budget of one selects (no cluster fits it)."""
import pytest
import torch

from paper_2502_05431_b200 import libape
from paper_2502_05431_b200 import workloads as wl
from tests.gpu_util import compare, gpu_attend, handle, kernels_in_order, oracle_attend

pytestmark = pytest.mark.gpu


def _ordinary(b, mode, **kw):
    handle().set_sm_budget(1)
    try:
        out, lse, n = gpu_attend(b, mode, **kw)
    finally:
        handle().set_sm_budget(0)
    assert n == 2
    return out, lse


def _kernels(b, mode, **how):
    dev = b.to("cuda:0")
    plan = handle().attend_plan(H_q=b.H_q, H_kv=b.H_kv, d=b.d, k_pool=dev.k_pool, v_pool=dev.v_pool, q=dev.q, out=torch.zeros_like(dev.q),
                                requests=b.requests, mode=mode, **how)
    plan.attend(b.T, b.S, plan.alloc_workspace())
    torch.cuda.synchronize()
    return plan.last_kernels()


@pytest.mark.parametrize("H_q,H_kv,d", [(32, 8, 128), (16, 1, 128), (8, 8, 64), (4, 1, 64), (2, 1, 128), (16, 8, 64)])
@pytest.mark.parametrize("n_req,ctx,l_P,l_k,gap", [(1, [64], 0, 1, 0), (1, [], 5, 1, 0), (2, [1, 63, 65, 200], 70, 3, 2), (3, [400, 7], 64, 64, 0),
                                                   (7, [129], 1, 130, 1)])
def test_decode(H_q, H_kv, d, n_req, ctx, l_P, l_k, gap):
    b = wl.make_batch(H_q=H_q, H_kv=H_kv, d=d, l_P=l_P, ctx_lens=[ctx] * n_req, l_q=1, l_k=l_k, capacity=l_k + 200, gap=gap, seed=41,
                      T=0.8, S=0.7, name="cluster")
    assert _kernels(b, libape.APE_DECODE) == 1
    for extra in (0, 1, 63, 200):
        out, lse, _ = gpu_attend(b, libape.APE_DECODE, kv_extra=extra)
        ref_o, ref_lse = _ordinary(b, libape.APE_DECODE, kv_extra=extra)
        # the same products and sums in another order, rounded to bf16 (2^-9 of the value) on both sides
        assert (out.float() - ref_o.float()).abs().max() <= 2 ** -7 * max(1.0, ref_o.float().abs().max().item())
        assert (lse - ref_lse).abs().max() < 1e-4
        for r, rq in enumerate(b.requests):
            ref = oracle_attend(b, r, l_k=l_k + extra)
            sl = slice(rq.q_start, rq.q_start + 1)
            compare(out[sl], ref.out.float(), f"req {r} extra {extra}")
            assert (lse[sl].double() - ref.lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("H_q,H_kv", [(3, 3), (4, 2), (8, 2), (16, 2), (32, 2)])
@pytest.mark.parametrize("lens", [[15, 17, 64], [128, 1, 79]])
def test_decode_query_heads_per_kv_head(H_q, H_kv, d, lens):
    """1, 2, 4, 8 query heads to a KV head are the columns of the products (8: all of them), 16 their rows; slices of 16 tokens that end
    inside, at the edge and before; both forms of the step."""
    b = wl.make_batch(H_q=H_q, H_kv=H_kv, d=d, l_P=33, ctx_lens=[lens, lens[:1]], l_q=1, l_k=5, capacity=70, gap=1, seed=51, T=0.8, S=0.7, name="heads")
    for extra in (0, 11, 12, 65):
        out, lse, n = gpu_attend(b, libape.APE_DECODE, kv_extra=extra)
        assert n == 1
        for got, got_lse in ((out, lse), _ordinary(b, libape.APE_DECODE, kv_extra=extra)):
            for r in range(2):
                ref = oracle_attend(b, r, l_k=5 + extra)
                compare(got[r:r + 1], ref.out.float(), f"req {r} extra {extra}")
                assert (got_lse[r:r + 1].double() - ref.lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("n_req,n_ctx,kernels", [(1, 10, 1), (1, 20, 2), (2, 10, 1), (2, 20, 2)])
def test_decode_on_both_sides_of_the_line(n_req, n_ctx, kernels):
    """The largest block of a cluster may have three tiles more than the ordinary form's: 5 against 3 and 9 against 5 tiles for one request (148 SMs)."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the split is that of 148 SMs")
    b = wl.make_batch(H_q=32, H_kv=8, d=128, l_P=32, ctx_lens=[[256] * n_ctx] * n_req, l_q=1, l_k=65, seed=42, T=0.8, S=0.7, name="line")
    out, lse, n = gpu_attend(b, libape.APE_DECODE)
    assert n == kernels
    for r in range(n_req):
        ref = oracle_attend(b, r)
        compare(out[r:r + 1], ref.out.float(), f"req {r}")
        assert (lse[r:r + 1].double() - ref.lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("n_req,lens,budget,kernels", [(1, [3000], 0, 1), (3, [64, 200, 1, 130], 0, 1), (3, [64, 200, 1, 130], 2, 3), (9, [640], 0, 1),
                                                       (9, [640], 2, 3), (33, [100, 700], 2, 3), (70, [129], 0, 3), (70, [129], 3, 3), (2, [], 0, 1)])
def test_shared_contexts_read_by_every_request_or_once(n_req, lens, budget, kernels):
    """A shared batch whose requests read the (few) contexts themselves (a cluster each), and, under an SM budget, the same batch with one
    pass over them."""
    b = wl.share_contexts(wl.make_batch(H_q=32, H_kv=8, d=128, l_P=7, ctx_lens=[lens] * n_req, l_q=1, l_k=3, capacity=90, gap=2, seed=43, T=0.8,
                                        S=0.7, name="shared"))
    handle().set_sm_budget(budget)
    try:
        out, lse, n = gpu_attend(b, libape.APE_DECODE, shared=True, kv_extra=70)
    finally:
        handle().set_sm_budget(0)
    assert n == kernels
    for r in (0, n_req // 2, n_req - 1):
        ref = oracle_attend(b, r, l_k=73)
        compare(out[r:r + 1], ref.out.float(), f"req {r}")
        assert (lse[r:r + 1].double() - ref.lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("n_req,n_ctx,length,gap,kernels", [(8, 120, 8, 3, 3), (8, 120, 8, 0, 2), (2, 120, 8, 3, 2), (4, 60, 129, 1, 3), (4, 30, 128, 0, 2), (3, 120, 16, 3, 2)])
def test_shared_contexts_of_short_spans(n_req, n_ctx, length, gap, kernels):
    """Spans that touch are one span; with gaps between them each is a tile of its own, for every request that reads it itself."""
    b = wl.share_contexts(wl.make_batch(H_q=32, H_kv=8, d=128, l_P=7, ctx_lens=[[length] * n_ctx] * n_req, l_q=1, l_k=3, gap=gap, seed=46, T=0.8,
                                        S=0.7, name="spans"))
    assert _kernels(b, libape.APE_DECODE, shared=True) == kernels
    out, lse, _ = gpu_attend(b, libape.APE_DECODE, shared=True)
    for r in (0, n_req - 1):
        ref = oracle_attend(b, r)
        compare(out[r:r + 1], ref.out.float(), f"req {r}")
        assert (lse[r:r + 1].double() - ref.lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("H_q,H_kv,d", [(32, 8, 128), (4, 1, 64), (16, 1, 128), (8, 8, 64)])
@pytest.mark.parametrize("n_req,ctx,l_P,l_q,l_k,gap", [(1, [], 0, 1, 1, 0), (1, [64] * 4, 16, 16, 16, 0), (2, [1, 130, 200], 70, 9, 140, 2),
                                                       (1, [900], 128, 33, 33, 0), (1, [129] * 3, 5, 129, 129, 1)])
def test_prefill(H_q, H_kv, d, n_req, ctx, l_P, l_q, l_k, gap):
    b = wl.make_batch(H_q=H_q, H_kv=H_kv, d=d, l_P=l_P, ctx_lens=[ctx] * n_req, l_q=l_q, l_k=l_k, gap=gap, seed=44, T=0.8, S=0.7, name="short")
    out, lse, n = gpu_attend(b, libape.APE_PREFILL)
    assert n == 1 or (H_q, ctx) == (4, [900])                  # (33 rows of four heads over nine tiles: the ordinary form)
    ref_o, ref_lse = _ordinary(b, libape.APE_PREFILL)
    compare(out, ref_o.float(), "cluster against ordinary")
    assert (lse - ref_lse).abs().max() < 1e-3
    for r, rq in enumerate(b.requests):
        ref = oracle_attend(b, r)
        sl = slice(rq.q_start, rq.q_start + rq.q_len)
        compare(out[sl], ref.out.float(), f"req {r}")
        assert (lse[sl].double() - ref.lse).abs().max().item() < 2e-3


# (query heads, contexts, rows) that the line between the forms sends to the ordinary one on 148 SMs
_ORDINARY_SHARES = {(4, 3, 32), (4, 5, 13), (4, 5, 32), (4, 9, 32), (4, 12, 1), (4, 12, 3), (4, 12, 13), (4, 12, 32), (16, 5, 13), (16, 9, 13),
                    (16, 12, 3), (16, 12, 13), (16, 12, 32)}


@pytest.mark.parametrize("H_q,H_kv,d", [(4, 1, 128), (16, 2, 64), (8, 8, 128)])
@pytest.mark.parametrize("n_ctx", [0, 1, 2, 3, 5, 9, 12])
@pytest.mark.parametrize("l_q", [1, 3, 13, 32])
def test_prefill_shares_of_rows(H_q, H_kv, d, n_ctx, l_q):
    """Every block of a cluster merges a share of the rows: rows that do not divide by the blocks, fewer rows than blocks, blocks without a
    partial, clusters of two to sixteen.  Against the ordinary form (the same products and sums in another order, rounded to bf16, 2^-9 of
    the value, on both sides) and the oracle; 13 of the 84 calls take the ordinary form themselves."""
    b = wl.make_batch(H_q=H_q, H_kv=H_kv, d=d, l_P=20, ctx_lens=[[130] * n_ctx], l_q=l_q, gap=1, seed=47, T=0.8, S=0.7, name="shares")
    out, lse, n = gpu_attend(b, libape.APE_PREFILL)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert n == (2 if (H_q, n_ctx, l_q) in _ORDINARY_SHARES else 1)
    ref_o, ref_lse = _ordinary(b, libape.APE_PREFILL)
    assert (out.float() - ref_o.float()).abs().max() <= 2 ** -7 * max(1.0, ref_o.float().abs().max().item())
    assert (lse - ref_lse).abs().max() < 1e-4
    ref = oracle_attend(b, 0)
    compare(out, ref.out.float(), "shares")
    assert (lse.double() - ref.lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("H_q,H_kv,l_q,lens,size", [
    (16, 4, 32, [[130] * 4, [130] * 4], 10),               # 128 rows, ten blocks of a tile: shares of 13 rows, the last of 11
    (16, 4, 32, [[130, 130, 130, 60], [130]], 9),          # nine blocks: shares of 15, rows from eight others fill what there is; four blocks, five idle
    (16, 4, 32, [[130] * 3, []], 8),                       # eight blocks, and two and six idle ones
    (32, 8, 32, [[130] * 4], 10), (28, 7, 20, [[130] * 7], 16)])       # (sixteen: 80 rows at most)
def test_prefill_full_row_blocks_in_large_clusters(H_q, H_kv, l_q, lens, size, d):
    """As many rows as a row block has in the clusters whose shares of them fill the space for rows from other blocks."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the split is that of 148 SMs")
    b = wl.make_batch(H_q=H_q, H_kv=H_kv, d=d, l_P=20, ctx_lens=lens, l_q=l_q, gap=1, seed=47, T=0.8, S=0.7, name="full")
    dev = b.to("cuda:0")
    plan = handle().attend_plan(H_q=H_q, H_kv=H_kv, d=d, k_pool=dev.k_pool, v_pool=dev.v_pool, q=dev.q, out=torch.zeros_like(dev.q),
                                requests=b.requests, mode=libape.APE_PREFILL)
    ws = plan.alloc_workspace()
    assert kernels_in_order(lambda: plan.attend(b.T, b.S, ws), grids=True) == [("attn", size * H_kv * len(lens))]
    out, lse, _ = gpu_attend(b, libape.APE_PREFILL)
    ref_o, ref_lse = _ordinary(b, libape.APE_PREFILL)
    assert (out.float() - ref_o.float()).abs().max() <= 2 ** -7 * max(1.0, ref_o.float().abs().max().item())
    assert (lse - ref_lse).abs().max() < 1e-4
    for r, rq in enumerate(b.requests):
        ref = oracle_attend(b, r)
        sl = slice(rq.q_start, rq.q_start + rq.q_len)
        compare(out[sl], ref.out.float(), f"req {r}")
        assert (lse[sl].double() - ref.lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("mode,l_q", [(libape.APE_DECODE, 1), (libape.APE_PREFILL, 20)])
def test_weights_that_are_no_numbers(mode, l_q, d):
    """A partial whose sum of weights is no positive number counts as empty, with a merge kernel or without: a head with NaN in its query
    gets zeros, and NaN in a key leaves no NaN behind."""
    b = wl.make_batch(H_q=8, H_kv=2, d=d, l_P=40, ctx_lens=[[300, 64, 65]], l_q=l_q, l_k=l_q + 3, seed=48, T=0.8, S=0.7, name="nan")
    assert _kernels(b, mode) == 1
    clean = gpu_attend(b, mode)[0]
    b.q[l_q - 1, 3] = float("nan")
    (out, lse, _), (ref_o, ref_lse) = gpu_attend(b, mode), _ordinary(b, mode)
    assert (out[l_q - 1, 3] == 0).all() and (ref_o[l_q - 1, 3] == 0).all()
    assert lse[l_q - 1, 3] == ref_lse[l_q - 1, 3] == float("-inf")
    out[l_q - 1, 3] = clean[l_q - 1, 3]
    assert torch.equal(out, clean)
    for s in (b.requests[0].ctx[1][0], b.requests[0].prefix[0]):
        b.k_pool[s, 1] = float("nan")
        assert torch.isfinite(gpu_attend(b, mode)[0].float()).all() and torch.isfinite(_ordinary(b, mode)[0].float()).all()


@pytest.mark.parametrize("mode,l_q", [(libape.APE_DECODE, 1), (libape.APE_PREFILL, 20)])
def test_scaling_beyond_the_range(mode, l_q):
    """S so large that the context's log-sum-exp is infinite: row and log-sum-exp are both no number, not one of them."""
    b = wl.make_batch(H_q=8, H_kv=2, d=64, l_P=40, ctx_lens=[[300]], l_q=l_q, seed=49, T=0.8, S=3e38, name="scale")
    for out, lse in (gpu_attend(b, mode)[:2], _ordinary(b, mode)):
        assert torch.isnan(out.float()).all() and torch.isnan(lse).all()


@pytest.mark.parametrize("H_q,H_kv,d,n_ctx,length,l_q,kernels", [
    (32, 8, 128, 10, 256, 64, 1), (16, 1, 128, 1, 512, 8, 1), (16, 1, 128, 1, 513, 8, 2),      # one row block of 128 rows: six tiles, seven
    (16, 1, 128, 1, 1200, 1, 1), (16, 1, 128, 1, 1281, 1, 2), (4, 1, 64, 1, 3000, 40, 2),      # of 16 rows: 12 and 13 tiles
    (16, 4, 128, 1, 2300, 16, 1), (16, 4, 128, 1, 3000, 8, 1), (16, 4, 128, 1, 3000, 32, 2),   # four row blocks: 10 partials, 13 of 32 and of 128 rows
])
def test_prefill_takes_clusters_where_they_are_faster(H_q, H_kv, d, n_ctx, length, l_q, kernels):
    """Large clusters merge slowly: only for several row blocks of few rows, small ones wherever the tiles fit (148 SMs)."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the split is that of 148 SMs")
    b = wl.make_batch(H_q=H_q, H_kv=H_kv, d=d, l_P=64, ctx_lens=[[length] * n_ctx], l_q=l_q, seed=47, T=0.8, S=0.7, name="line")
    assert _kernels(b, libape.APE_PREFILL) == kernels
    out, lse, _ = gpu_attend(b, libape.APE_PREFILL)
    ref = oracle_attend(b, 0)
    compare(out, ref.out.float(), "line")
    assert (lse.double() - ref.lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("budget", [2, 40, 147])
@pytest.mark.parametrize("mode,l_q,shared", [(libape.APE_DECODE, 1, False), (libape.APE_DECODE, 1, True), (libape.APE_PREFILL, 16, False)])
def test_no_clusters_under_a_budget(budget, mode, l_q, shared):
    """A cluster waits for free SMs in one part of the chip, and the kernel that the budget is for takes some of every part."""
    b = wl.make_batch(H_q=4, H_kv=1, d=128, l_P=8, ctx_lens=[[64] * 4], l_q=l_q, seed=45, T=0.8, S=0.7, name="budget")
    assert _kernels(b, mode, shared=shared) == 1
    handle().set_sm_budget(budget)
    try:
        assert _kernels(b, mode, shared=shared) == 2
        out, lse, _ = gpu_attend(b, mode, shared=shared)
    finally:
        handle().set_sm_budget(0)
    ref = oracle_attend(b, 0)
    compare(out, ref.out.float(), f"budget {budget}")
    assert (lse.double() - ref.lse).abs().max().item() < 2e-3
