"""What orders the parts of the library that run side by side: the warps of a block, the kernels of a call, calls on one stream."""
import pytest
import torch

from paper_2502_05431_b200 import libape
from paper_2502_05431_b200 import workloads as wl
from tests.gpu_util import handle
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
