"""Timed cases of the APE attention path: the calls that a serving or evaluation program makes, over the range it makes them.

Every case is one operation of the public interface (paper_2502_05431_b200.libape):

  prefill   attention of the query rows over [prefix | contexts | causal query segment]; `form` is the plain one (Eq. 5),
            the per-context one (Eq. 11-12) or a two-level context tree
  decode    one new token per request over the same cache, `step` tokens after planning
  shared    the same for a batch of requests over ONE set of cached contexts
  encode    pre-caching attention of every context (block-diagonal, behind the shared prefix)
  rope      rotary embedding with position re-use, fused with the write of K, V and Q to their rows

The shapes are those of paper_2502_05431_b200.workloads (tiny, 10 x 256, RAG with 20 contexts of 512 to 1536 tokens, many-shot
with 500 x 256 tokens = 128K) and, for the drawn cases, the ranges between and around them with the head layouts of the tests.
"""
import random

import torch

from paper_2502_05431_b200 import libape
from paper_2502_05431_b200 import workloads as wl

LLAMA = dict(H_q=32, H_kv=8, d=128)
TINY = dict(H_q=4, H_kv=1, d=64)
HEADS = [(32, 8, 128), (32, 8, 128), (32, 8, 128), (8, 2, 64), (4, 1, 64), (8, 8, 128), (16, 1, 128), (16, 4, 128)]
THETA = 500000.0


def _case(name, op, *, form="eq5", l_P=64, n_req=1, n_ctx=10, len_lo=256, len_hi=256, len_seed=0, l_q=1, l_k=0, step=0, gap=0,
          lse=False, T=0.9, S=0.9, H_q=32, H_kv=8, d=128):
    c = dict(op=op, form=form, l_P=l_P, n_req=n_req, n_ctx=n_ctx, len_lo=len_lo, len_hi=len_hi, len_seed=len_seed, l_q=l_q,
             l_k=l_k or l_q, step=step, gap=gap, lse=lse, T=T, S=S, H_q=H_q, H_kv=H_kv, d=d)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # A short question over four small passages on one KV head of a small model: latency of a launch-sized call.
        _case("prefill_tiny_d64", "prefill", l_P=16, n_ctx=4, len_lo=64, len_hi=64, l_q=16, lse=True, T=0.8, S=0.9, **TINY),
        # A 64-token question over ten retrieved passages: the ordinary interactive call, first token.
        _case("prefill_10x256", "prefill", l_P=32, l_q=64),
        # Four users' questions over twenty ragged documents each: the ordinary RAG batch.
        _case("prefill_rag_4x20", "prefill", n_req=4, n_ctx=20, len_lo=512, len_hi=1536, l_q=128, S=0.8),
        # Many-shot prompt of 128K cached tokens, 256 query rows: the longest first token.
        _case("prefill_500x256", "prefill", n_ctx=500, l_q=256),
        # The same prompt with the scaling factor on every context's own mass.
        _case("prefill_per_context_500x256", "prefill", form="per_context", n_ctx=500, l_q=256),
        # One user's next token over ten passages: latency of the smallest decode step.
        _case("decode_1x10x256", "decode", l_P=32, l_k=65, step=17),
        # The next token of a RAG batch (ragged documents).
        _case("decode_rag_4x20", "decode", n_req=4, n_ctx=20, len_lo=512, len_hi=1536, l_k=129, step=40, S=0.8),
        # The next token of sixteen users with 128K cached tokens each: the largest decode batch.
        _case("decode_16x500x256", "decode", n_req=16, n_ctx=500, l_k=257, step=128),
        # The next token of sixteen users who ask about the same 128K cached tokens.
        _case("shared_16x500x256", "shared", n_req=16, n_ctx=500, l_k=257, step=128),
        # Caching ten passages, as they come in.
        _case("encode_10x256", "encode", l_P=32, lse=True),
        # Caching a many-shot corpus of 128K tokens.
        _case("encode_500x256", "encode", n_ctx=500),
        # Rotating and writing K, V and Q of that corpus to its cache rows, in front of the encode.
        _case("rope_500x256", "rope", n_ctx=500),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    while True:
        op = rng.choice(["prefill", "prefill", "prefill", "decode", "decode", "shared", "encode", "encode", "rope"])
        H_q, H_kv, d = rng.choice(HEADS)
        form = rng.choice(["eq5", "eq5", "per_context", "tree"]) if op == "prefill" else \
            rng.choice(["eq5", "eq5", "eq5", "per_context"]) if op == "decode" else "eq5"
        n_ctx = _log_int(rng, 1, 500)
        mean = _log_int(rng, 16, 2048)
        spread = rng.choice([0.0, 0.5])
        n_req = 1 if op in ("encode", "rope") else _log_int(rng, 1, 32 if op == "shared" else 16 if op == "decode" else 4)
        l_q = _log_int(rng, 1, 512) if op == "prefill" else 1
        c = _case(None, op, form=form, l_P=rng.choice([0, 16, 32, 64, 100, 128, 130]), n_req=n_req, n_ctx=n_ctx,
                  len_lo=max(1, int(mean * (1 - spread))), len_hi=max(1, int(mean * (1 + spread))),
                  len_seed=rng.randrange(1 << 20), l_q=l_q, l_k=l_q + (rng.choice([0, 0, 63, 256]) if op != "prefill" else rng.choice([0, 0, 70])),
                  step=rng.choice([0, 1, 17, 100]) if op in ("decode", "shared") else 0, gap=rng.choice([0, 0, 3]),
                  lse=op != "rope" and rng.random() < 0.3, T=rng.choice([0.5, 0.8, 0.9, 1.0]), S=rng.choice([0.6, 0.8, 0.9, 1.0]),
                  H_q=H_q, H_kv=H_kv, d=d)
        w = work(c)
        # no case costs more than the largest listed ones: 128K cached tokens a request, a third of their arithmetic, half of their
        # bytes; the per-context decode step keeps a partial per context, so it is drawn with fewer of them
        if n_ctx * mean <= 131072 and w["flops"] <= 2e11 and w["bytes"] <= 4e9 and (op != "decode" or form == "eq5" or n_ctx <= 100):
            return c


def _lens(c):
    rng = random.Random(c["len_seed"])
    return [[rng.randint(c["len_lo"], c["len_hi"]) for _ in range(c["n_ctx"])] for _ in range(c["n_req"])]


def _tree(c):
    """Every fifth node a document (top level, carries S), the nodes behind it its sections."""
    return [[-1 if i % 5 == 0 else i - i % 5 for i in range(c["n_ctx"])] for _ in range(c["n_req"])]


class State:
    pass


_handles = {}


def _handle():
    dev = torch.cuda.current_device()
    if dev not in _handles:
        _handles[dev] = libape.Handle(dev)
    return _handles[dev]


def _batch(c, seed):
    dev = f"cuda:{torch.cuda.current_device()}"
    lens = _lens(c)
    # the requests of a shared batch keep only their own prefix and query segment; the contexts are request 0's
    lens_made = lens if c["op"] != "shared" else [lens[0]] + [[] for _ in range(c["n_req"] - 1)]
    b = wl.make_batch(H_q=c["H_q"], H_kv=c["H_kv"], d=c["d"], l_P=c["l_P"], ctx_lens=lens_made, l_q=c["l_q"], l_k=c["l_k"],
                      capacity=c["l_k"] + (256 if c["op"] in ("decode", "shared") else 0), seed=1000 * (int(seed) + 1), T=c["T"], S=c["S"],
                      head_scale=c["n_ctx"] >= 100, gap=c["gap"], with_encode_q=c["op"] in ("encode", "rope"), device=dev)
    if c["op"] == "shared":
        for r in b.requests[1:]:
            r.ctx = list(b.requests[0].ctx)
    return b


def prepare(case, seed):
    b = _batch(case, seed)
    s = State()
    s.op, s.b, s.case = case["op"], b, case
    heads = dict(H_q=b.H_q, H_kv=b.H_kv, d=b.d)
    s.lse = None
    if s.op == "encode":
        s.out = torch.zeros_like(b.q_enc)
        if case["lse"]:
            s.lse = torch.zeros((b.q_enc.shape[0], b.H_q), dtype=torch.float32, device=b.q.device)
        r = b.requests[0]
        s.plan = _handle().encode_plan(**heads, k_pool=b.k_pool, v_pool=b.v_pool, q=b.q_enc, out=s.out, prefix=r.prefix, ctx=r.ctx, lse=s.lse)
    elif s.op == "rope":
        # the packed, unrotated rows of prefix, contexts and question; their rows in the cache; K, V and Q land there
        r = b.requests[0]
        s.src = (b.k_pool, b.v_pool, b.q_enc)
        s.dst = tuple(torch.zeros_like(t) for t in s.src)
        s.plan = libape.RopePlan(_handle(), b.d, THETA, libape.rope_runs_for_request(r))
    else:
        s.out = torch.zeros_like(b.q)
        if case["lse"]:
            s.lse = torch.zeros((b.q.shape[0], b.H_q), dtype=torch.float32, device=b.q.device)
        s.plan = _handle().attend_plan(**heads, k_pool=b.k_pool, v_pool=b.v_pool, q=b.q, out=s.out, requests=b.requests,
                                       mode=libape.APE_PREFILL if s.op == "prefill" else libape.APE_DECODE, lse=s.lse,
                                       per_context=case["form"] == "per_context", shared=s.op == "shared",
                                       tree=(_tree(case), None) if case["form"] == "tree" else None)
        s.ws = s.plan.alloc_workspace()
    return s


def run(state):
    s, c = state, state.case
    if s.op == "encode":
        s.plan.encode_contexts()
    elif s.op == "rope":
        for src, dst, rotate in zip(s.src, s.dst, (True, False, True)):
            s.plan.write(src, dst, rotate)
        return {"k": s.dst[0], "v": s.dst[1], "q": s.dst[2]}
    else:
        s.plan.attend(c["T"], c["S"], s.ws, kv_extra=c["step"])
    return {"out": s.out} if s.lse is None else {"out": s.out, "lse": s.lse}


def work(case):
    c, lens = case, _lens(case)
    row_q, row_kv = 2 * c["H_q"] * c["d"], 2 * 2 * c["H_kv"] * c["d"]          # bytes of a row of Q or O; of K and V together
    per_pair = 4 * c["d"] * c["H_q"]                                           # multiply-adds of q.k and p.v, all heads
    if c["op"] == "rope":
        rows = c["l_P"] + sum(lens[0]) + c["l_k"]
        return {"bytes": 2 * rows * (row_q + row_kv), "flops": 6 * rows * (c["H_q"] + c["H_kv"]) * c["d"] // 2}
    if c["op"] == "encode":
        rows = sum(lens[0])
        pairs = sum(n * c["l_P"] + n * (n + 1) // 2 for n in lens[0])
        return {"bytes": 2 * rows * row_q + (c["l_P"] + rows) * row_kv, "flops": pairs * per_pair}
    if c["op"] == "shared":
        own = c["l_P"] + c["l_k"] + c["step"]
        return {"bytes": 2 * c["n_req"] * row_q + (sum(lens[0]) + c["n_req"] * own) * row_kv,
                "flops": c["n_req"] * (sum(lens[0]) + own) * per_pair}
    l_k = c["l_k"] + c["step"]
    seen = c["l_q"] * l_k - c["l_q"] * (c["l_q"] - 1) // 2
    keys = sum(c["l_P"] + sum(ln) + l_k for ln in lens)
    pairs = sum(c["l_q"] * (c["l_P"] + sum(ln)) + seen for ln in lens)
    return {"bytes": 2 * c["n_req"] * c["l_q"] * row_q + keys * row_kv, "flops": pairs * per_pair}


def tolerance(case):
    # bf16 results of fp32 sums over bf16 weights: 2.4e-3 against 64 bits is seen for attention, 1.7e-3 for the rotation (one
    # rounding of the result); rows with few keys have the largest single differences
    return {"rel": 7e-3 if case["op"] == "rope" else 1e-2, "max": 0.25}


# ---- the same results in 64 bits, from plain torch operations -----------------------------------------------------------------

def _take(pool, span, g):
    return pool[span[0]:span[0] + span[1], g].double()


def _attend64(c, b, r, parent, scaled, out, lse):
    """Eq. 5 (parent None) or the tree form of one request: `parent[i]`, `scaled[i]` of context i."""
    G, scale, T, S = b.H_q // b.H_kv, b.d ** -0.5, c["T"], c["S"]
    rq, n, l_k = b.requests[r], b.requests[r].q_len, b.requests[r].query_kv[1] + c["step"]
    kq = (rq.query_kv[0], l_k)
    ctx = [x for x in rq.ctx]
    idx = torch.cat([torch.arange(s, s + ln, device=b.q.device) for s, ln in ctx]) if ctx else torch.empty(0, dtype=torch.long, device=b.q.device)
    hidden = torch.arange(l_k, device=b.q.device)[None, :] > torch.arange(n, device=b.q.device)[:, None] + (l_k - n)
    for g in range(b.H_kv):
        q = b.q[rq.q_start:rq.q_start + n, g * G:(g + 1) * G].double().reshape(n * G, b.d)
        xo = torch.cat([q @ _take(b.k_pool, rq.prefix, g).T, (q @ _take(b.k_pool, kq, g).T).masked_fill(hidden.repeat_interleave(G, 0), -torch.inf)], 1) * scale
        vo = torch.cat([_take(b.v_pool, rq.prefix, g), _take(b.v_pool, kq, g)])
        xc = q @ b.k_pool[idx, g].double().T * (scale / T)
        if parent is None:
            xc += (S - 1) * torch.logsumexp(xc, 1, keepdim=True) if ctx else 0
        else:
            own = [torch.logsumexp(p, 1) for p in xc.split([ln for _, ln in ctx], 1)]
            mass, inside = [None] * len(ctx), [[o] for o in own]
            for i in reversed(range(len(ctx))):
                mass[i] = torch.logsumexp(torch.stack(inside[i]), 0)
                if parent[i] >= 0:
                    inside[parent[i]].append(S * mass[i] if scaled[i] else mass[i])
            bias = [None] * len(ctx)
            for i in range(len(ctx)):
                bias[i] = (bias[parent[i]] if parent[i] >= 0 else 0) + ((S - 1) * mass[i] if scaled[i] else torch.zeros_like(mass[i]))
            for part, o in zip(xc.split([ln for _, ln in ctx], 1), bias):
                part += o[:, None]
        total = torch.logaddexp(torch.logsumexp(xo, 1), torch.logsumexp(xc, 1)) if ctx else torch.logsumexp(xo, 1)
        o = (xo - total[:, None]).exp_() @ vo
        if ctx:
            o += xc.sub_(total[:, None]).exp_() @ b.v_pool[idx, g].double()
        out[rq.q_start:rq.q_start + n, g * G:(g + 1) * G] = o.reshape(n, G, b.d)
        lse[rq.q_start:rq.q_start + n, g * G:(g + 1) * G] = total.reshape(n, G)


def _encode64(b, out, lse):
    G, scale, rq = b.H_q // b.H_kv, b.d ** -0.5, b.requests[0]
    spread = lambda pool, span: pool[span[0]:span[0] + span[1]].double().transpose(0, 1).repeat_interleave(G, 0)  # noqa: E731
    kp, vp = spread(b.k_pool, rq.prefix), spread(b.v_pool, rq.prefix)
    for s, n in rq.ctx:
        q = b.q_enc[s:s + n].double().transpose(0, 1)
        hidden = torch.ones((n, n), dtype=torch.bool, device=q.device).triu(1)
        x = torch.cat([q @ kp.transpose(1, 2), (q @ spread(b.k_pool, (s, n)).transpose(1, 2)).masked_fill(hidden, -torch.inf)], 2) * scale
        total = torch.logsumexp(x, 2, keepdim=True)
        out[s:s + n] = ((x - total).exp() @ torch.cat([vp, spread(b.v_pool, (s, n))], 1)).transpose(0, 1)
        lse[s:s + n] = total[:, :, 0].T


def _rope64(b):
    rq = b.requests[0]
    dst = [torch.zeros(t.shape, dtype=torch.float64, device=t.device) for t in (b.k_pool, b.v_pool, b.q_enc)]
    longest, src = max([ln for _, ln in rq.ctx], default=0), 0
    runs = [(rq.prefix, 0)] + [(s, rq.prefix[1]) for s in rq.ctx] + [(rq.query_kv, rq.prefix[1] + longest)]
    freq = THETA ** (-2.0 * torch.arange(b.d // 2, dtype=torch.float64, device=b.q.device) / b.d)
    for (to, n), pos in runs:
        phi = (pos + torch.arange(n, dtype=torch.float64, device=b.q.device))[:, None, None] * freq
        cos, sin = phi.cos(), phi.sin()
        for t, d, rotate in zip((b.k_pool, b.v_pool, b.q_enc), dst, (True, False, True)):
            x = t[src:src + n].double()
            lo, hi = x.chunk(2, -1)
            d[to:to + n] = torch.cat([lo * cos - hi * sin, hi * cos + lo * sin], -1) if rotate else x
        src += n
    return {"k": dst[0], "v": dst[1], "q": dst[2]}


def exact(case, seed):
    b = _batch(case, seed)
    if case["op"] == "rope":
        return _rope64(b)
    like = b.q_enc if case["op"] == "encode" else b.q
    out = torch.zeros(like.shape, dtype=torch.float64, device=like.device)
    lse = torch.zeros(like.shape[:2], dtype=torch.float64, device=like.device)
    if case["op"] == "encode":
        _encode64(b, out, lse)
    else:
        for r in range(case["n_req"]):
            if case["form"] == "eq5":
                _attend64(case, b, r, None, None, out, lse)
            else:
                parent = _tree(case)[r] if case["form"] == "tree" else [-1] * case["n_ctx"]
                _attend64(case, b, r, parent, [p < 0 for p in parent], out, lse)
    return {"out": out, "lse": lse} if case["lse"] else {"out": out}
