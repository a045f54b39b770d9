"""GPU parity of the shared-context decode plan (a batch of queries over ONE set of cached contexts, read once) against
the fp64 oracle, request by request, through the C ABI."""
import pytest
import torch

from paper_2502_05431_b200 import libape, workloads as wl
from tests.gpu_util import handle, gpu_attend, kernels_in_order, oracle_attend, compare

pytestmark = pytest.mark.gpu
LLAMA = dict(H_q=32, H_kv=8, d=128)


def _check(b, once, kv_extra=0, lse_tol=2e-3):
    """once: the contexts are read once for the batch (rest, context pass, merge); else every request reads them itself."""
    out, lse, n = gpu_attend(b, libape.APE_DECODE, shared=True, kv_extra=kv_extra)
    assert n == 3 if once else n < 3
    for r, rq in enumerate(b.requests):
        ref = oracle_attend(b, r, l_k=(rq.query_kv[1] + kv_extra) if kv_extra else None)
        compare(out[rq.q_start:rq.q_start + 1], ref.out.float(), f"{b.name} req {r} O")
        d = (lse[rq.q_start:rq.q_start + 1].double() - ref.lse).abs().max().item()
        assert d < lse_tol, f"{b.name} req {r}: LSE error {d}"
    return out


@pytest.mark.parametrize("kw,n_req,once", [
    (dict(**LLAMA, l_P=16, ctx_lens=[64, 200, 1, 130], l_k=5, T=0.9, S=0.9), 3, False),
    (dict(**LLAMA, l_P=16, ctx_lens=[9600, 200, 1, 1300], l_k=5, T=0.9, S=0.9), 3, True),
    (dict(**LLAMA, l_P=7, ctx_lens=[300], l_k=66, T=0.6, S=1.2, gap=2), 16, False),
    (dict(**LLAMA, l_P=7, ctx_lens=[1300], l_k=66, T=0.6, S=1.2, gap=2), 16, True),
    (dict(H_q=8, H_kv=8, d=64, l_P=3, ctx_lens=[100, 100], l_k=9, T=0.9, S=0.5), 5, False),        # G = 1, d = 64
    (dict(H_q=8, H_kv=8, d=64, l_P=3, ctx_lens=[3300, 2900], l_k=9, T=0.9, S=0.5), 5, True),
    (dict(H_q=16, H_kv=1, d=128, l_P=64, ctx_lens=[256] * 3, l_k=65, T=1.1, S=0.9), 20, False),    # G = 16: two row blocks
    (dict(H_q=16, H_kv=1, d=128, l_P=64, ctx_lens=[256] * 28, l_k=65, T=1.1, S=0.9), 20, True),
    (dict(**LLAMA, l_P=4, ctx_lens=[], l_k=3, T=0.9, S=0.9), 2, False),                            # no contexts at all
    (dict(**LLAMA, l_P=900, ctx_lens=[], l_k=3, T=0.9, S=0.9), 16, False),                         # (the rest and the merge alone)
    (dict(**LLAMA, l_P=0, ctx_lens=[129], l_k=1, T=0.8, S=0.7), 70, True),                         # 70 x 4 rows: two row blocks, ragged
    (dict(**LLAMA, l_P=5, ctx_lens=[100], l_k=2, T=0.9, S=0.9), 32, False),
    (dict(**LLAMA, l_P=300, ctx_lens=[100], l_k=2, T=0.9, S=0.9), 32, True),                       # 128 rows exactly, one tile: one half idle
    (dict(**LLAMA, l_P=5, ctx_lens=[100, 700], l_k=2, T=0.9, S=0.9), 33, True),                    # 132 rows: one 256-row block again
    (dict(**LLAMA, l_P=9, ctx_lens=[128 * 5], l_k=2, T=0.7, S=0.8), 9, False),
    (dict(**LLAMA, l_P=9, ctx_lens=[128 * 21], l_k=2, T=0.7, S=0.8), 9, True),                     # an odd number of whole tiles
])
def test_shared_context_decode(kw, n_req, once):
    lens = kw.pop("ctx_lens")
    b = wl.share_contexts(wl.make_batch(ctx_lens=[lens] + [lens if not once else []] * (n_req - 1), l_q=1, seed=21, name="shared", **kw))
    _check(b, once)


@pytest.mark.parametrize("length,once", [(256, False), (2048, True)])
def test_shared_plan_agrees_with_the_per_request_plan_and_grows(length, once):
    b = wl.share_contexts(wl.make_batch(**LLAMA, l_P=32, ctx_lens=[[length] * 6] + [[]] * 3, l_q=1, l_k=40, capacity=60, seed=22,
                                        T=0.9, S=0.9, name="shared_grow"))
    for t in (0, 1, 20):
        out = _check(b, once, kv_extra=t)
        ref, _, _ = gpu_attend(b, libape.APE_DECODE, kv_extra=t)                # ordinary decode plan on the same requests
        assert (out.float() - ref.float()).abs().max().item() <= 2e-2


def test_shared_plan_rejects_requests_that_do_not_share():
    b = wl.make_batch(**LLAMA, l_P=8, ctx_lens=[[64], [64]], l_q=1, l_k=4, seed=23)     # two different context sets
    dev = torch.device("cuda:0")
    q, k, v = b.q.to(dev), b.k_pool.to(dev), b.v_pool.to(dev)
    out = torch.empty_like(q)
    with pytest.raises(libape.ApeError) as e:
        handle().attend_plan(H_q=32, H_kv=8, d=128, k_pool=k, v_pool=v, q=q, out=out, requests=b.requests,
                             mode=libape.APE_DECODE, shared=True)
    assert e.value.code == -1
    s = wl.share_contexts(b)
    s.requests[1].q_start = 0                                                          # rows not consecutive
    with pytest.raises(libape.ApeError) as e:
        handle().attend_plan(H_q=32, H_kv=8, d=128, k_pool=k, v_pool=v, q=q, out=out, requests=s.requests,
                             mode=libape.APE_DECODE, shared=True)
    assert e.value.code == -1


def test_shared_decode_at_the_benchmark_size_sampled_requests():
    """16 requests over one set of 500 x 256 cached context tokens behind a 64-token prefix, the shape bench.py times;
    the oracle checks sampled requests at the first and a late decode step."""
    lens = [[256] * 500] + [[]] * 15                      # only request 0 owns contexts in the pool; the others borrow them
    b = wl.share_contexts(wl.make_batch(**LLAMA, l_P=64, ctx_lens=lens, l_q=1, l_k=257, capacity=257 + 255, seed=31,
                                        T=0.9, S=0.9, name="shared_128k"))
    for t in (0, 255):
        out, lse, n = gpu_attend(b, libape.APE_DECODE, shared=True, kv_extra=t)
        assert n == 3
        for r in (0, 7, 15):
            rq = b.requests[r]
            ref = oracle_attend(b, r, l_k=rq.query_kv[1] + t)
            compare(out[r:r + 1], ref.out.float(), f"shared 128K step {t} req {r}")
            assert (lse[r:r + 1].double() - ref.lse).abs().max().item() < 2e-3


@pytest.mark.parametrize("H_q,H_kv,d,n_req,n_ctx,capacity,first", [
    (32, 8, 128, 16, 2000, 64, "attn"), (32, 8, 128, 16, 2000, 65, "decode"),        # alternating halves: 1.73 and 2.6 tiles per SM
    (16, 1, 128, 24, 6000, 320, "attn"), (16, 1, 128, 24, 6000, 321, "decode"),      # 384 rows: 0.97 and 1.14
    (8, 2, 64, 32, 4096, 400, "attn"),                                               # heads of 64
])
def test_order_of_a_shared_step(H_q, H_kv, d, n_req, n_ctx, capacity, first):
    """The per-request rest goes in front of the context pass where it is long enough to be worth it (148 SMs)."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the line is drawn in tiles per SM")
    b = wl.share_contexts(wl.make_batch(H_q=H_q, H_kv=H_kv, d=d, l_P=7, ctx_lens=[[n_ctx]] + [[]] * (n_req - 1), l_q=1, l_k=30, capacity=capacity, seed=34,
                                        T=0.9, S=0.9, name="order"))
    dev = b.to("cuda:0")
    out = torch.zeros_like(dev.q)
    plan = handle().attend_plan(H_q=H_q, H_kv=H_kv, d=d, k_pool=dev.k_pool, v_pool=dev.v_pool, q=dev.q, out=out, requests=b.requests,
                                mode=libape.APE_DECODE, shared=True)
    ws = plan.alloc_workspace()
    assert kernels_in_order(lambda: plan.attend(b.T, b.S, ws, kv_extra=3)) == [first, {"attn": "decode", "decode": "attn"}[first], "merge"]
    for r in (0, n_req - 1):
        compare(out[r:r + 1].cpu(), oracle_attend(b, r, l_k=33).out.float(), f"{first} first, req {r}")
