"""What orders the parts of the library that run side by side: the warps of a block, the kernels of a call, calls on one stream."""
import ctypes as C

import pytest
import torch

from paper_2502_05431_b200 import libape
from paper_2502_05431_b200 import workloads as wl
from tests.gpu_util import compare, handle, oracle_attend
from tests.test_gpu_parity import _check_encode

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("l_P", [0, 64])
@pytest.mark.parametrize("heads", [dict(H_q=32, H_kv=8, d=128), dict(H_q=8, H_kv=2, d=64)])
@pytest.mark.parametrize("lens", [[64] * 200, [64, 33, 32, 96, 256] * 40])
def test_encode_stages_two_row_blocks_at_a_time(l_P, heads, lens):
    """Row blocks of one or two tiles with full halves, which leave through their Q buffer: a half may stage a row block while the
    other half's previous one has not been sent.  Every row against the oracle, then the same bits again and again."""
    b = wl.make_batch(**heads, l_P=l_P, ctx_lens=[lens], l_q=1, seed=60, with_encode_q=True, name="staged")
    _check_encode(b)
    dev = torch.device("cuda:0")
    rq = b.requests[0]
    q, k, v = b.q_enc.to(dev), b.k_pool.to(dev), b.v_pool.to(dev)
    outs = [torch.zeros_like(q) for _ in range(2)]
    plans = [handle().encode_plan(H_q=b.H_q, H_kv=b.H_kv, d=b.d, k_pool=k, v_pool=v, q=q, out=o, prefix=rq.prefix, ctx=rq.ctx) for o in outs]
    plans[0].encode_contexts()
    for _ in range(30):
        outs[1].zero_()
        plans[1].encode_contexts()
        assert torch.equal(outs[0], outs[1])
    assert handle().get_status() == 0


EARLY_AND_LONG = """
extern "C" __global__ void early_and_long() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long t0 = clock64();
    while (clock64() - t0 < 2800000000ll) {}
}
"""


@pytest.mark.parametrize("op", ["prefill", "per_context", "decode", "encode"])
def test_time_limit_of_waits_starts_after_the_kernel_before(op):
    """A kernel (any library's) that lets the next one in early and then runs for longer than the limit of a bounded wait (2^31
    cycles): what a call waits for meanwhile is that kernel, and it must not count as a copy or product that never came."""
    b = wl.make_batch(H_q=32, H_kv=8, d=128, l_P=30, ctx_lens=[[256, 70, 1]], l_q=1 if op == "decode" else 70, l_k=75, seed=61, T=0.8, S=0.9,
                      with_encode_q=True, name="late").to("cuda:0")
    rq, heads = b.requests[0], dict(H_q=32, H_kv=8, d=128, k_pool=b.k_pool, v_pool=b.v_pool)
    q = b.q_enc if op == "encode" else b.q
    out = torch.zeros_like(q)
    if op == "encode":
        plan = handle().encode_plan(**heads, q=q, out=out, prefix=rq.prefix, ctx=rq.ctx)
        launch = plan.encode_contexts
    else:
        plan = handle().attend_plan(**heads, q=q, out=out, requests=b.requests, per_context=op == "per_context",
                                    mode=libape.APE_DECODE if op == "decode" else libape.APE_PREFILL)
        ws = plan.alloc_workspace()
        launch = lambda: plan.attend(b.T, b.S, ws)  # noqa: E731
    launch()
    first = out.clone()
    out.zero_()
    before = torch.cuda._compile_kernel(EARLY_AND_LONG, "early_and_long")
    before(grid=(1, 1, 1), block=(32, 1, 1), args=[])
    launch()
    torch.cuda.synchronize()
    assert handle().get_status() == 0
    assert torch.equal(out, first)


def _same_with_and_without_waits(launches, bufs):
    """Chains of 1, 2, ... calls, each reading the buffer that the one before it wrote: the same bits with a synchronisation behind
    every call and with nothing at all between two calls."""
    start = bufs[0].clone()
    for n in range(1, len(launches) + 1):
        ends = []
        for wait in (True, False):
            bufs[0].copy_(start)
            bufs[1].zero_()
            torch.cuda.synchronize()
            for launch in launches[:n]:
                launch()
                if wait:
                    torch.cuda.synchronize()
            torch.cuda.synchronize()
            ends.append([x.clone() for x in bufs])
        assert not torch.isnan(ends[0][n % 2].float()).any()
        assert torch.equal(ends[0][0], ends[1][0]) and torch.equal(ends[0][1], ends[1][1]), f"{n} calls"
        assert not torch.equal(ends[0][0], ends[0][1])
    assert handle().get_status() == 0


@pytest.mark.parametrize("mode,l_q,n_req,longest,l_P,kernels", [
    (libape.APE_DECODE, 1, 4, 256, 30, (1, 1)),            # clusters
    (libape.APE_DECODE, 1, 4, 6000, 30, (2, 3)),           # shared: context pass, rest, merge
    (libape.APE_DECODE, 1, 24, 700, 30, (2, 3)),           # shared: rest, context pass beside it (alternating halves), merge
    (libape.APE_DECODE, 1, 40, 300, 30, (2, 3)),           # the same with 160 rows
    (libape.APE_PREFILL, 64, 1, 256, 30, (1,)), (libape.APE_PREFILL, 200, 1, 700, 900, (2,)),
    (libape.APE_PREFILL, 200, 1, 18000, 30, (2,)),         # siblings and 30 tiles a group: the attention kernel is launched in order
])
def test_calls_that_feed_each_other(mode, l_q, n_req, longest, l_P, kernels):
    """The output of a call is the query of the next, all calls share one workspace, and no kernel of another library stands between
    them: what a kernel reads too early is an older query, partial or bias.  All plan kinds, each call over contexts of its own."""
    b = wl.make_batch(H_q=32, H_kv=8, d=128, l_P=l_P, ctx_lens=[[longest, 70, 130, 64] * 12] * n_req, l_q=l_q, l_k=l_q + 5, seed=62, T=0.7, S=0.8,
                      name="chain", device="cuda:0")
    b.v_pool *= 8                              # (large outputs, a high logit scale: a call's query decides its result)
    bufs = [b.q, torch.zeros_like(b.q)]
    forms = [dict(), dict(per_context=True), dict(tree=([[-1, 0, 0, 0]] * n_req, None))]
    if mode == libape.APE_DECODE:
        forms.append(dict(shared=True))
    plans = []
    for i in range(12):
        form = forms[i % len(forms)]
        ctx = [r.ctx[4 * i:4 * i + 4] for r in b.requests]
        reqs = [wl.Request(r.q_start, r.q_len, r.prefix, ctx[0 if form.get("shared") else j], r.query_kv, r.query_kv_capacity)
                for j, r in enumerate(b.requests)]
        plans.append(handle().attend_plan(H_q=32, H_kv=8, d=128, k_pool=b.k_pool, v_pool=b.v_pool, q=bufs[i % 2], out=bufs[(i + 1) % 2],
                                          requests=reqs, mode=mode, softmax_scale=0.5, **form))
    ws = torch.empty(max(p.workspace_bytes for p in plans), dtype=torch.uint8, device="cuda:0")
    _same_with_and_without_waits([lambda p=p: p.attend(b.T, b.S, ws) for p in plans], bufs)
    assert plans[0].last_launches() == kernels[0]          # Eq. 5
    if mode == libape.APE_DECODE:
        assert plans[3].last_launches() == kernels[1]      # shared contexts


def test_encode_and_prefill_that_feed_each_other():
    b = wl.make_batch(H_q=32, H_kv=8, d=128, l_P=64, ctx_lens=[[256] * 8], l_q=1, l_k=9, seed=63, T=0.7, S=0.8, with_encode_q=True,
                      name="chain_encode").to("cuda:0")
    b.v_pool *= 8
    rq, heads = b.requests[0], dict(H_q=32, H_kv=8, d=128, k_pool=b.k_pool, v_pool=b.v_pool, softmax_scale=0.5)
    bufs = [torch.nan_to_num(b.q_enc), torch.zeros_like(b.q_enc)]
    plans = []
    for i in range(10):
        io = dict(q=bufs[i % 2], out=bufs[(i + 1) % 2])
        if i % 2 == 0:
            plans.append(handle().encode_plan(**heads, **io, prefix=rq.prefix, ctx=rq.ctx))
        else:                                  # the rows of every context, over all the contexts but that one
            reqs = [wl.Request(s, n, rq.prefix, [c for c in rq.ctx if c[0] != s], (s, n), n) for s, n in rq.ctx]
            plans.append(handle().attend_plan(**heads, **io, requests=reqs, mode=libape.APE_PREFILL))
    ws = torch.empty(max(p.workspace_bytes for p in plans), dtype=torch.uint8, device="cuda:0")
    _same_with_and_without_waits([p.encode_contexts if i % 2 == 0 else lambda p=p: p.attend(b.T, b.S, ws) for i, p in enumerate(plans)], bufs)


@pytest.mark.parametrize("op", ["encode", "decode", "prefill", "per_context", "shared"])
def test_budget_leaves_the_other_sms_free(op):
    """A long call on one SM with another call queued behind it: a call on a second stream, which needs whole SMs, runs meanwhile on
    the ones that the budget leaves.  (None of the calls waits for another one's result.)"""
    n = 4000 if op == "encode" else 60000
    b = wl.make_batch(H_q=32, H_kv=8, d=128, l_P=64, ctx_lens=[[n], [64]], l_q=1, l_k=9, seed=64, T=0.8, S=0.9, with_encode_q=True,
                      name="budget", device="cuda:0")
    rq, rq1 = b.requests
    reqs = [rq] if op != "shared" else [rq, wl.Request(rq1.q_start, 1, rq1.prefix, rq.ctx, rq1.query_kv, rq1.query_kv_capacity)]
    heads = dict(H_q=32, H_kv=8, d=128, k_pool=b.k_pool, v_pool=b.v_pool)
    form = dict(per_context=op == "per_context", shared=op == "shared")
    handle().set_sm_budget(1)
    try:
        if op == "encode":
            long = handle().encode_plan(**heads, q=b.q_enc, out=torch.zeros_like(b.q_enc), prefix=rq.prefix, ctx=rq.ctx)
        else:
            mode = libape.APE_DECODE if op in ("decode", "shared") else libape.APE_PREFILL
            long = handle().attend_plan(**heads, q=b.q, out=torch.zeros_like(b.q), requests=reqs, mode=mode, **form)
    finally:
        handle().set_sm_budget(0)
    ws = [long.alloc_workspace()]
    run_long = long.encode_contexts if op == "encode" else lambda: long.attend(b.T, b.S, ws[0])
    other = wl.make_batch(H_q=32, H_kv=8, d=128, l_P=64, ctx_lens=[[64] * 40], l_q=64, l_k=64, seed=65, T=0.8, S=0.9, name="beside",
                          device="cuda:0")
    after, beside = [handle().attend_plan(H_q=32, H_kv=8, d=128, k_pool=other.k_pool, v_pool=other.v_pool, q=other.q,
                                          out=torch.zeros_like(other.q), requests=other.requests, mode=libape.APE_PREFILL) for _ in range(2)]
    ws += [after.alloc_workspace(), beside.alloc_workspace()]
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    run_long(), after.attend(0.8, 0.9, ws[1]), beside.attend(0.8, 0.9, ws[2])       # (first launches load code)
    torch.cuda.synchronize()
    assert long.last_launches() == {"encode": 1, "shared": 3, "per_context": 4}.get(op, 2)
    with torch.cuda.stream(s1):
        run_long()
        after.attend(0.8, 0.9, ws[1])
        done = s1.record_event()
    with torch.cuda.stream(s2):
        beside.attend(0.8, 0.9, ws[2])
    s2.synchronize()
    assert not done.query(), "the call beside it only ran once the long call had ended"
    torch.cuda.synchronize()
    assert handle().get_status() == 0


def test_decode_plans_of_other_head_layouts_leave_a_plan_usable():
    """The shared memory that a decode launch asks for depends on G; the kernel's limit is one per process and must not follow the plan
    made last (nor an allocation-free call)."""
    plans = []
    for H_q, H_kv in ((32, 8), (16, 1), (8, 8), (16, 8)):
        b = wl.make_batch(H_q=H_q, H_kv=H_kv, d=128, l_P=20, ctx_lens=[[300, 5]], l_q=1, l_k=9, seed=66, T=0.8, S=0.9, name=f"G{H_q // H_kv}")
        dev = b.to("cuda:0")
        out = torch.zeros_like(dev.q)
        plan = handle().attend_plan(H_q=H_q, H_kv=H_kv, d=128, k_pool=dev.k_pool, v_pool=dev.v_pool, q=dev.q, out=out, requests=b.requests,
                                    mode=libape.APE_DECODE)
        plans.append((b, dev, plan, out, plan.alloc_workspace()))
    for b, dev, plan, out, ws in plans + plans[:1]:
        plan.attend(b.T, b.S, ws)
        compare(out.cpu(), oracle_attend(b, 0).out.float(), b.name)
    b, dev, _, out, _ = plans[1]
    libape.decode_noalloc(H_q=16, H_kv=1, d=128, k_pool=dev.k_pool, v_pool=dev.v_pool, q=dev.q, out=out, requests=b.requests, T=b.T, S=b.S,
                          want_status=True)
    b, dev, plan, out, ws = plans[0]
    plan.attend(b.T, b.S, ws)
    compare(out.cpu(), oracle_attend(b, 0).out.float(), b.name)


def test_a_failed_launch_is_not_blamed_on_a_later_call():
    """Calls that fail on the host (here: on a stream whose capture has been invalidated, where every launch is refused) leave nothing
    behind that makes a later, good call report an error."""
    rt = C.CDLL("libcudart.so.12")
    b = wl.make_batch(H_q=32, H_kv=8, d=128, l_P=20, ctx_lens=[[64]], l_q=4, l_k=9, seed=67, T=0.8, S=0.9, name="blame").to("cuda:0")
    out = torch.zeros_like(b.q)
    make = lambda: handle().attend_plan(H_q=32, H_kv=8, d=128, k_pool=b.k_pool, v_pool=b.v_pool, q=b.q, out=out, requests=b.requests,  # noqa: E731
                                        mode=libape.APE_PREFILL)
    plan, rope = make(), libape.RopePlan(handle(), 128, 500000.0, [(0, 0, 20, 0)])
    ws, dst = plan.alloc_workspace(), torch.zeros_like(b.k_pool)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    assert rt.cudaStreamBeginCapture(C.c_void_p(s.cuda_stream), 0) == 0
    try:
        with pytest.raises(libape.ApeError):
            make()                                                 # allocates: not allowed, and ends the capture's validity
        with pytest.raises(libape.ApeError) as e:
            plan.attend(b.T, b.S, ws, stream=s)
        assert e.value.code == -7
    finally:
        graph = C.c_void_p()
        assert rt.cudaStreamEndCapture(C.c_void_p(s.cuda_stream), C.byref(graph)) != 0 and not graph.value
        rt.cudaGetLastError()
    rope.write(b.k_pool, dst, False)
    part = [torch.zeros(1, 4, 32, 128, device="cuda:0"), torch.zeros(1, 4, 32, device="cuda:0")]
    libape.merge_shards(handle(), H_q=32, H_kv=8, d=128, o_ctx_all=part[0], lse_ctx_all=part[1], o_oth=part[0][0], lse_oth=part[1][0], S=1.0,
                        out=out)
    plan.attend(b.T, b.S, ws)
    torch.cuda.synchronize()
    assert torch.equal(dst[:20], b.k_pool[:20]) and handle().get_status() == 0
