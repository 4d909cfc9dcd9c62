"""The work that a program has this framework do, as cases that can be timed and compared.

A case is one pass of a serving program through the public entry points: a decoded token through
a few MoE layers, a batch of streams, a verification batch, a prefill chunk.  Shapes are those of
``synth/configs.py`` (hidden 256 / 2048 / 2816, 8 - 128 experts, top-2 / top-8, intermediate
512 / 768 / 1408, Q8_0 and Q4_0) and a ragged one.  Expert weights are normal values quantised
as GGUF files hold them; routes are Zipf-popular expert sets planted through the logit bias, as
in the repository's benchmark, or the router's own choice where there is no bias.

Keys of a case: api ("device", "host" or "noalloc"); L layers, H hidden, E experts, k chosen, I
intermediate, q GGUF type (8: Q8_0, 2: Q4_0), T tokens a call, steps (calls of every layer in one
pass), S slots a layer (E: everything resident before the pass), zipf and reuse of the routes
(planted False: the router chooses), cold (the pass starts with an empty cache), order of the
cache accesses, graph (the calls are captured once and replayed, as a decode loop does).
"""
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_2607_09686_gb300 as mf

Q8, Q4 = mf.Q8_0, mf.Q4_0
BASE = dict(api="device", L=1, H=2048, E=128, k=8, I=768, q=Q8, T=1, steps=1, S=128, zipf=1.2, reuse=0.0,
            planted=True, cold=False, order=0, graph=False)


def _case(name, **kw):
    return dict(BASE, name=name, **kw)


def listed():
    return [
        # the smallest call: one decoded token, one small layer, the router's own choice
        _case("decode_tiny_q8", H=256, E=8, k=2, I=512, S=8, planted=False),
        # one decoded token through four layers whose experts are all resident, replayed as a graph
        _case("decode_q8", L=4, E=64, S=64, zipf=1.1, reuse=0.6, graph=True),
        # the same through the host-buffer entry point (pinned x, bias and y), call by call, 4-bit experts
        _case("decode_q4_host", api="host", L=4, E=64, S=64, q=Q4, zipf=1.1),
        # 16 tokens in a row through four layers from an empty cache of 35 % of the experts
        _case("decode_stream_q8", L=4, E=64, S=22, steps=16, zipf=1.1, reuse=0.6, cold=True, graph=True),
        # the expert FFN alone, on weights that the caller holds
        _case("ffn_noalloc_q8", api="noalloc", E=8, S=8, planted=False),
        # a model whose sizes are multiples of 32 and of nothing larger
        _case("decode_ragged_q4", L=2, H=1440, E=60, k=5, I=544, q=Q4, S=60, zipf=0.8),
        # a verification batch of speculative decoding: five rows a call
        _case("verify_q8", T=5, zipf=1.2),
        # 64 decode streams, everything resident
        _case("streams64_q8", H=2816, I=1408, T=64, zipf=1.0),
        # 64 decode streams on a cache of 15 %: several waves a call, resident experts first
        _case("streams64_waves_q4", q=Q4, T=64, S=19, zipf=1.0, order=1),
        # a prefill chunk of odd length, everything resident
        _case("prefill_1000_q8", E=64, S=64, T=1000, zipf=0.8),
        # a full prefill chunk, everything resident
        _case("prefill_4096_q4", q=Q4, T=4096),
        # the same chunk on an empty cache of 15 %: the experts arrive wave by wave
        _case("prefill_4096_q4_cold", q=Q4, T=4096, S=19, cold=True),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _payload_bytes(c):
    return 3 * c["H"] * c["I"] // 32 * (34 if c["q"] == Q8 else 18)


def draw(rng):
    while True:
        c = dict(BASE)
        c["q"] = rng.choice((Q8, Q4))
        kind = rng.choice(("decode", "decode", "stream", "host", "noalloc", "small", "streams", "prefill", "prefill"))
        step = 128 if kind == "prefill" or rng.random() < 0.4 else 32
        c["H"] = step * max(1, round(_log(rng, 256, 2816) / step))
        c["I"] = step * max(1, round(_log(rng, 128, 1408) / step))
        c["E"] = round(_log(rng, 8, 128))
        c["k"] = min(c["E"], rng.choice((1, 2, 3, 4, 5, 6, 7, 8, 8, 8, 8)))
        c["zipf"] = rng.choice((0.0, 0.8, 1.0, 1.1, 1.2))
        c["S"] = c["E"]
        partial = max(c["k"], int(c["E"] * rng.choice((0.15, 0.25, 0.35, 0.5, 0.65))))
        if kind in ("decode", "stream"):
            c["L"] = rng.randint(1, 4)
            c["graph"] = rng.random() < 0.5
            c["reuse"] = rng.choice((0.0, 0.6, 0.8))
            if kind == "stream":
                c.update(steps=rng.randint(2, 16), S=partial, cold=True)
        elif kind == "host":
            c.update(api="host", L=rng.randint(1, 4), T=rng.choice((1, 1, 1, 3)))
        elif kind == "noalloc":
            c.update(api="noalloc", E=c["k"], S=c["k"], planted=False)
        else:
            lo, hi = {"small": (2, 16), "streams": (16, 128), "prefill": (256, 4096)}[kind]
            c.update(T=round(_log(rng, lo, hi)), order=rng.choice((0, 1)))
            if rng.random() < 0.4:
                c.update(S=partial, cold=kind == "prefill")
        if _payload_bytes(c) * c["E"] * c["L"] > 1.4e9 or c["T"] * c["k"] * c["H"] * c["I"] > 4096 * 8 * 2048 * 768:
            continue
        return c


def _quantise(w, q):
    """Values in blocks of 32 along the last axis -> GGUF block bytes (uint8, [..., blocks, 34 or 18])."""
    b = w.reshape(*w.shape[:-1], -1, 32)
    if q == Q8:
        d = (b.abs().amax(-1, keepdim=True) / 127).half()
        n = torch.round(b / d.float().clamp_min(1e-8)).clamp_(-127, 127).to(torch.int8)
        codes = n.view(torch.uint8)
    else:
        m = torch.take_along_dim(b, b.abs().argmax(-1, keepdim=True), -1)
        d = (m / -8).half()
        n = (torch.round(b / torch.where(d == 0, 1, d.float())) + 8).clamp_(0, 15).to(torch.uint8)
        codes = n[..., :16] | (n[..., 16:] << 4)
    return torch.cat((d.view(torch.uint8), codes), -1)


def _dequantise(blocks, q):
    """GGUF block bytes -> the values they stand for, in 64 bits."""
    d = blocks[..., :2].contiguous().view(torch.float16).double()
    c = blocks[..., 2:].contiguous()
    n = c.view(torch.int8).double() if q == Q8 else torch.cat((c & 15, c >> 4), -1).double() - 8
    return (d * n).flatten(-2)


def _experts(c, seed, layer):
    """One layer's experts on the GPU: gate [E, I, H / 32, B], up the same, down [E, H, I / 32, B]."""
    g = torch.Generator("cuda").manual_seed(seed * 1009 + layer + 1)
    shapes = ((c["I"], c["H"]), (c["I"], c["H"]), (c["H"], c["I"]))
    return [torch.stack([_quantise(torch.randn(s, device="cuda", generator=g) * (1.0 / math.sqrt(s[1])), c["q"])
                         for _ in range(c["E"])]) for s in shapes]


def _inputs(c, seed):
    """Per layer: router weights [E, H], x [steps * T, H], bias [steps * T, E] or None (on the GPU)."""
    g = torch.Generator("cuda").manual_seed(seed * 7919 + 17)
    n, E, k = c["steps"] * c["T"], c["E"], c["k"]
    out = []
    for _ in range(c["L"]):
        wr = torch.randn(E, c["H"], device="cuda", generator=g) * 0.02
        x = torch.randn(n, c["H"], device="cuda", generator=g)
        bias = None
        if c["planted"]:
            # k draws without replacement, expert of rank r with weight (r + 1)^-zipf, ranks permuted
            p = -c["zipf"] * torch.log(torch.arange(1, E + 1, device="cuda", dtype=torch.float32))
            p = p[torch.randperm(E, device="cuda", generator=g)]
            u = torch.rand(n, E, device="cuda", generator=g).clamp_(1e-12, 1 - 1e-7)
            sets = (p - torch.log(-torch.log(u))).topk(k, 1).indices
            if c["reuse"] > 0:  # a token keeps the previous one's set with this probability
                new = torch.rand(n, device="cuda", generator=g) >= c["reuse"]
                at = torch.where(new, torch.arange(n, device="cuda"), 0).cummax(0).values
                sets = sets[at]
            bias = torch.zeros(n, E, device="cuda")
            bias.scatter_(1, sets, (16 + 0.5 * (k - torch.arange(k, device="cuda", dtype=torch.float32))).expand(n, k))
        out.append((wr, x, bias))
    return out


def _noalloc_inputs(c, seed):
    g = torch.Generator("cuda").manual_seed(seed * 7919 + 17)
    x = torch.randn(c["H"], device="cuda", generator=g)
    return x, torch.softmax(torch.randn(c["k"], device="cuda", generator=g), 0)


def _slots(c, gate, up, down):
    """The caller-held slots of mf_expert_ffn_noalloc, as mawforge.h lays them out."""
    def up16(v):
        return (v + 15) // 16 * 16

    def up256(v):
        return (v + 255) // 256 * 256

    H, I, E = c["H"], c["I"], c["E"]
    flip = 128 if c["q"] == Q8 else 0
    codes = [(t[..., 2:] ^ flip).flatten(2) for t in (gate, up, down)]
    scales = [t[..., :2].flatten(2) for t in (gate, up, down)]
    o_gs = 2 * codes[0].shape[2]
    o_us = o_gs + up16(2 * (H // 32))
    rs_gu, rs_d = up16(o_us + 2 * (H // 32)), up16(codes[2].shape[2] + 2 * (I // 32))
    d_off = up256(I * rs_gu)
    slot = torch.zeros(E, up256(d_off + H * rs_d), dtype=torch.uint8, device="cuda")
    gu = slot[:, :I * rs_gu].view(E, I, rs_gu)
    for t, at in ((codes[0], 0), (codes[1], codes[0].shape[2]), (scales[0], o_gs), (scales[1], o_us)):
        gu[:, :, at:at + t.shape[2]] = t
    dn = slot[:, d_off:d_off + H * rs_d].view(E, H, rs_d)
    for t, at in ((codes[2], 0), (scales[2], codes[2].shape[2])):
        dn[:, :, at:at + t.shape[2]] = t
    return slot


class _State:
    """A context with its pack, and the buffers of a pass."""

    ctx = graph = None

    def close(self):
        self.graph = None
        if self.ctx:
            mf.mf_destroy(self.ctx)
            self.ctx = None

    def __del__(self):
        self.close()


def _calls(s):
    fwd = mf.mf_moe_forward_host if s.host else mf.mf_moe_forward
    if s.cold:
        mf.mf_reset(s.ctx)
    for layer, x, wr, bias, y, idx, w in s.args:
        fwd(s.ctx, layer, x, wr, bias, s.T, y, idx, w)


def prepare(case, seed):
    c = case
    s = _State()
    s.T, s.cold, s.host = c["T"], c["cold"], c["api"] == "host"
    s.model = mf.Model(c["L"], c["H"], c["E"], c["k"], c["I"], c["q"])
    if c["api"] == "noalloc":
        s.slots = _slots(c, *_experts(c, seed, 0))
        s.x, s.g = _noalloc_inputs(c, seed)
        s.y = torch.empty(c["H"], device="cuda")
        return s
    plan = mf.mf_plan(s.model, mf.PlanReq(100.0 * c["S"] / c["E"], 1 << 62, 0, 0, c["T"], 0))
    s.ctx = mf.mf_create(s.model, plan, 0)
    with ThreadPoolExecutor(16) as pool:
        for layer in range(c["L"]):
            packs = torch.cat([t.flatten(1) for t in _experts(c, seed, layer)], 1).cpu().numpy()
            list(pool.map(lambda e: mf.mf_pack_put(s.ctx, layer, e, packs[e]), range(c["E"])))
    if c["order"]:
        mf.mf_access_order(s.ctx, c["order"])
    L, n, T, k = c["L"], c["steps"] * c["T"], c["T"], c["k"]
    ins = _inputs(c, seed)
    if s.host:
        def place(t):
            return None if t is None else t.cpu().pin_memory()
    else:
        def place(t):
            return t
    s.ins = [(wr, place(x), place(b)) for wr, x, b in ins]
    s.y = place(torch.empty(L, n, c["H"], device="cuda"))
    s.idx = place(torch.empty(L, n, k, dtype=torch.int32, device="cuda"))
    s.w = place(torch.empty(L, n, k, device="cuda"))
    s.args = []
    for t in range(0, n, T):
        r = slice(t, t + T)
        for l, (wr, x, b) in enumerate(s.ins):
            s.args.append((l, x[r], wr, None if b is None else b[r], s.y[l, r], s.idx[l, r], s.w[l, r]))
    if c["S"] == c["E"]:  # earlier calls have made every expert resident
        for first in range(0, c["E"], k):
            b = torch.zeros(T, c["E"], device="cuda")
            b[:, first:first + k] = 64.0
            for l, (wr, x, _) in enumerate(ins):
                mf.mf_moe_forward(s.ctx, l, x[:T], wr, b, T, s.y[l, :T] if not s.host else torch.empty_like(x[:T]))
            torch.cuda.synchronize()
    if c["graph"]:
        _calls(s)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            _calls(s)
        s.graph = graph
    return s


def run(state):
    s = state
    if s.ctx is None:
        mf.mf_expert_ffn_noalloc(s.model, s.slots, s.g, s.x, s.y)
        return s.y
    if s.graph is not None:
        s.graph.replay()
    else:
        _calls(s)
    return {"y": s.y, "idx": s.idx, "w": s.w}


def _distinct(c):
    """Distinct experts of one call and of one layer's whole pass, of a fixed draw of the routes."""
    if c["api"] == "noalloc" or (c["T"] == 1 and c["steps"] == 1):
        return c["k"], c["k"]
    r = np.random.RandomState(11)
    n, T = c["steps"] * c["T"], c["T"]
    p = -c["zipf"] * np.log(np.arange(1, c["E"] + 1)) if c["planted"] else np.zeros(c["E"])
    sets = np.argsort(-(p + r.gumbel(size=(n, c["E"]))), 1)[:, :c["k"]]
    at = np.maximum.accumulate(np.where(r.rand(n) >= c["reuse"], np.arange(n), 0))
    sets = sets[at]
    call = np.mean([len(np.unique(sets[t:t + T])) for t in range(0, n, T)])
    return float(call), float(len(np.unique(sets)))


def work(case):
    """Quantised weights of each call's distinct experts (and, from an empty cache or one too small
    for a call, their transfer into the slots), router weights, x, bias, y, indices and weights."""
    c = case
    call, whole = _distinct(c)
    calls, n = c["L"] * c["steps"], c["L"] * c["steps"] * c["T"]
    b = calls * call * _payload_bytes(c) + n * c["H"] * 8
    f = n * c["k"] * 6 * c["H"] * c["I"]
    if c["api"] == "noalloc":
        return {"bytes": b + 4 * c["k"], "flops": f}
    if c["S"] < c["E"]:
        moved = whole if c["cold"] else max(0.0, call - c["S"])
        b += c["L"] * moved * _payload_bytes(c)
    b += calls * c["E"] * c["H"] * 4 + n * (c["E"] * 4 * c["planted"] + c["k"] * 8)
    return {"bytes": b, "flops": f + n * 2 * c["E"] * c["H"]}


def tolerance(case):
    """About four times the error against exact(), measured over the listed and drawn cases: up to
    1e-6 where sums are 32-bit or exact integers, up to 1.8e-5 in chunks of 256 tokens and more,
    whose operands are pairs of bf16 values (16 bits)."""
    c = case
    pairs = c["T"] >= 256 and c["H"] % 128 == 0 and c["I"] % 128 == 0
    return {"rel": 8e-5} if pairs else {"rel": 4e-6}


def _ffn(x, gate, up, down):
    h = x @ gate.T
    return (h / (1 + torch.exp(-h)) * (x @ up.T)) @ down.T


def exact(case, seed):
    c = case
    if c["api"] == "noalloc":
        ex = [_dequantise(t, c["q"]) for t in _experts(c, seed, 0)]
        x, g = (t.double() for t in _noalloc_inputs(c, seed))
        return sum(g[j] * _ffn(x[None], ex[0][j], ex[1][j], ex[2][j])[0] for j in range(c["k"]))
    ys, ws = [], []
    for layer, (wr, x, bias) in enumerate(_inputs(c, seed)):
        x = x.double()
        z = (x @ wr.double().T).float()  # logits are the 32-bit rounding of the dot product
        z = (z if bias is None else z + bias)
        top = z.sort(dim=1, descending=True, stable=True)
        idx, w = top.indices[:, :c["k"]], torch.softmax(top.values[:, :c["k"]].double(), 1)
        gate, up, down = _experts(c, seed, layer)
        y = torch.zeros_like(x)
        for e in torch.unique(idx).tolist():
            t, j = torch.nonzero(idx == e, as_tuple=True)
            y.index_add_(0, t, w[t, j, None] * _ffn(x[t], *(_dequantise(m[e], c["q"]) for m in (gate, up, down))))
        ys.append(y)
        ws.append(w)
    return {"y": torch.stack(ys), "idx": None, "w": torch.stack(ws)}
