"""What orders the parts of the library that run side by side: the warps of a block, the kernels of a call, calls on one stream."""
import pytest
import torch

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
