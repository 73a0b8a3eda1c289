"""The work that a user of this library has it do, as cases that can be timed.

Three kinds of pass, all through `DmcCache`:

  generate  one request batch served: reset, the prompt compressed into every
            layer, then decode steps through the layers (one launch per layer,
            one launch for all layers, or each step's launches replayed from a
            CUDA graph). Returns every step's attention outputs and the slot
            counts (a step attends over every slot as updated by that step, so
            the outputs show the whole cache). The reset makes every pass do
            the same work.
  compress  a prompt node: reset, one layer's prompt compressed, all of its
            heads exported into dense buffers (to hand the cache to another
            process). Returns the buffers.
  attend    prompt attention of one layer, the prompt in one call or continued
            over several. Returns every token's output and the slot counts.

Inputs follow the repository's workloads: Gaussian k and v at scale 0.5, the
decision neuron k[0] away from its tie and negative (append) with probability
1/CR of its head, the importance neuron q[0] at scale 0.5; the other query
components have scale 2, so that scores spread by about one (a softmax that
picks among its slots). Prompt lengths and the heads' compression ratios follow
from the case alone, all values from the seed.
"""
import math

import torch

from paper_2403_09636_gb300 import DmcCache

_GOLDEN = 0.6180339887498949
_PAGE = 32


def _case(name, kind, **kw):
    c = {"name": name, "kind": kind, "mode": "layer", "layers": 1, "batch": 1, "q_heads": 32, "kv_heads": 32,
         "head_dim": 128, "dtype": "bf16", "prompt_lo": 2048, "prompt_hi": 2048, "parts": 1, "steps": 0,
         "cr_lo": 4.0, "cr_hi": 4.0, "window": 0}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest configuration, whole: 4 fp32 heads of dim 64, a 256-token prompt, 32 decode steps of
        # one layer (launches and latency)
        _case("tiny_f32", "generate", q_heads=4, kv_heads=4, head_dim=64, dtype="f32", prompt_lo=256, prompt_hi=256,
              steps=32, cr_lo=2.0, cr_hi=2.0),
        # one user's chat on the 7B shape: batch 1, each step's launches replayed from a CUDA graph
        _case("chat_7b_batch1", "generate", mode="graph", layers=8, steps=16),
        # batched serving on the 7B shape at 4x, one launch per layer and step
        _case("decode_7b_4x", "generate", layers=4, batch=32, steps=32),
        # the same on the 70B shape: 8 queries per KV head, 2x
        _case("decode_70b_gqa_2x", "generate", layers=2, batch=64, q_heads=64, kv_heads=8, prompt_lo=4096,
              prompt_hi=4096, steps=32, cr_lo=2.0, cr_hi=2.0),
        # mixed compression ratios per head, every decode step one launch over all layers
        _case("layers_7b_mixed", "generate", mode="layers", layers=4, batch=32, steps=16, cr_lo=1.0, cr_hi=8.0),
        # long ragged prompts with heavy-tailed ratios: mostly prompt compression, a few tokens answered
        _case("long_ragged", "generate", batch=8, prompt_lo=1024, prompt_hi=32768, steps=8, cr_lo=1.0, cr_hi=32.0),
        # the window-grouping approximation on the 7B shape
        _case("window12_7b_4x", "generate", layers=2, batch=32, steps=32, window=12),
        # a prompt node on the 7B shape: compress, then export every head
        _case("handover_7b_4x", "compress", batch=32),
        # prompt attention of one layer: 7B (one query per KV head) and 70B (groups of 8)
        _case("attend_7b_4x", "attend", batch=32),
        _case("attend_70b_gqa_2x", "attend", batch=16, q_heads=64, kv_heads=8, prompt_lo=4096, prompt_hi=4096,
              cr_lo=2.0, cr_hi=2.0),
        # a handful of short prompts of odd lengths, groups of 4: the latency of an interactive prompt
        _case("attend_short_ragged", "attend", batch=5, q_heads=32, kv_heads=8, prompt_lo=19, prompt_hi=700,
              cr_lo=1.0, cr_hi=8.0),
        # one long document, prefilled in four chunks that each continue the cache
        _case("attend_long_chunked", "attend", q_heads=64, kv_heads=8, prompt_lo=16384, prompt_hi=16384, parts=4,
              cr_lo=2.0, cr_hi=2.0),
    ]


def _cost(c):
    """About the microseconds of a pass, to keep drawn cases within the listed ones."""
    w = work(c)
    calls = c["layers"] * (c["steps"] + 2) + 4 * c["parts"]
    return w["bytes"] / 5e6 + w["flops"] / 5e8 + 10.0 * calls


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["generate", "generate", "generate", "compress", "attend", "attend"])
    hq, hkv = rng.choice([(32, 32), (40, 40), (64, 8), (32, 8), (16, 8), (8, 8)])
    c = _case("", kind, q_heads=hq, kv_heads=hkv, batch=spread(1, 64))
    del c["name"]
    hi = spread(24, 16384)
    c["prompt_hi"] = hi
    c["prompt_lo"] = hi if rng.random() < 0.4 else max(1, int(hi * rng.uniform(0.05, 0.9)))
    c["cr_lo"] = rng.choice([1.0, 2.0, 4.0])
    c["cr_hi"] = c["cr_lo"] * rng.choice([1.0, 1.0, 4.0, 8.0])
    if kind == "generate":
        c["mode"] = rng.choice(["layer", "layer", "layers", "graph"])
        c["layers"] = rng.randint(1, 4)
        c["steps"] = spread(2, 32)
        c["window"] = rng.choice([0, 0, 0, 12])
    if kind == "attend":
        c["parts"] = rng.choice([1, 1, 2, 3])
    else:
        c["head_dim"] = rng.choice([128, 128, 64])
        c["dtype"] = rng.choice(["bf16", "bf16", "bf16", "f32"])
    most = 0.9 * max(_cost(x) for x in listed())
    while _cost(c) > most:
        if c["batch"] > 1:
            c["batch"] = (c["batch"] + 1) // 2
        else:
            c["prompt_hi"] = max(24, c["prompt_hi"] // 2 + 1)
            c["prompt_lo"] = min(c["prompt_lo"], c["prompt_hi"])
    return c


# ---------------------------------------------------------------- sizes that follow from the case

def _lengths(c):
    """Prompt tokens of every sequence."""
    lo, hi = c["prompt_lo"], c["prompt_hi"]
    return [lo + int((hi - lo + 1) * ((0.5 + i * _GOLDEN) % 1.0)) for i in range(c["batch"])]


def _append_prob(c):
    """1 / CR of every (layer, KV head), CR spread between cr_lo and cr_hi over its logarithm."""
    L, H = c["layers"], c["kv_heads"]
    lo, hi = math.log(c["cr_lo"]), math.log(c["cr_hi"])
    return [[math.exp(-(lo + (hi - lo) * ((0.25 + (layer * H + h) * _GOLDEN) % 1.0))) for h in range(H)]
            for layer in range(L)]


def _slot_bound(n, p):
    """Slots that n tokens appended with probability p stay below."""
    return min(n, int(n * p + 6.0 * math.sqrt(n * p * (1.0 - p)) + 8))


def _part(n, parts, i):
    """Tokens [a, b) of part i of an n-token prompt."""
    return n * i // parts, n * (i + 1) // parts


def work(c):
    D, Hq, H = c["head_dim"], c["q_heads"], c["kv_heads"]
    es = 4 if c["dtype"] == "f32" else 2
    row = D * es
    lens, probs = _lengths(c), _append_prob(c)
    tokens = sum(lens)
    nbytes = flops = 0.0
    for layer in range(c["layers"]):
        ptot = sum(probs[layer])  # slots of one token over the heads
        nbytes += tokens * (2 * H * row + Hq * es)           # k, v and the importance neurons
        nbytes += tokens * ptot * (2 * row + 4)              # slots and z written
        if c["kind"] == "generate":
            slots = sum(n * ptot for n in lens)
            nbytes += c["steps"] * (slots * 2 * row + c["batch"] * (2 * Hq + 4 * H) * row)
            flops += c["steps"] * slots * (Hq // H) * 4.0 * D
        elif c["kind"] == "compress":
            cap = _export_cap(c)
            nbytes += tokens * ptot * (2 * row + 4)          # read back by the export
            nbytes += c["batch"] * H * cap * (2 * row + 4)   # the buffers written
        else:
            nbytes += 2.0 * tokens * Hq * row                # queries read, outputs written
            for n in lens:
                flops += 4.0 * D * (Hq // H) * (n * (n - 1) / 2.0 * ptot + n * H)
    return {"bytes": nbytes, "flops": flops}


def _export_cap(c):
    p = max(max(x) for x in _append_prob(c))
    return -(-_slot_bound(max(_lengths(c)), p) // _PAGE) * _PAGE


# ---------------------------------------------------------------- inputs

def _dtype(c):
    return torch.float32 if c["dtype"] == "f32" else torch.bfloat16


def _tokens(c, g, shape, probs, full_q):
    """q, k, v of tokens laid out as `shape` (probs: the heads' append probabilities, broadcast over it)."""
    dt, dev = _dtype(c), torch.device("cuda")
    H, Hq, D = c["kv_heads"], c["q_heads"], c["head_dim"]

    def normal(*s):
        return torch.randn(*s, generator=g, device=dev, dtype=dt)

    k = normal(*shape, H, D).mul_(0.5)
    v = normal(*shape, H, D).mul_(0.5)
    mag = torch.randn(*shape, H, generator=g, device=dev).abs_().add_(0.1).mul_(0.5)
    opens = torch.rand(*shape, H, generator=g, device=dev) < probs
    k[..., 0] = torch.where(opens, -mag, mag).to(dt)
    q0 = normal(*shape, Hq).mul_(0.5)
    if not full_q:
        return q0, k, v
    q = normal(*shape, Hq, D).mul_(2.0)
    q[..., 0] = q0
    return q, k, v


def _inputs(c, seed):
    """Prompts, a list over layers of lists over parts of (q, k, v, cu_seqlens, max length), and the decode
    steps' q, k, v as [steps, layers, batch, heads, head_dim]."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    lens, dev = _lengths(c), torch.device("cuda")
    probs = torch.tensor(_append_prob(c), dtype=torch.float32, device=dev)
    prompts = []
    for layer in range(c["layers"]):
        parts = []
        for i in range(c["parts"]):
            n = [b - a for a, b in (_part(x, c["parts"], i) for x in lens)]
            cu = torch.tensor([0] + n, dtype=torch.int64).cumsum(0).to(torch.int32).to(dev)
            parts.append((*_tokens(c, g, (sum(n),), probs[layer], c["kind"] == "attend"), cu, max(n)))
        prompts.append(parts)
    decode = None
    if c["steps"]:
        decode = _tokens(c, g, (c["steps"], c["layers"], c["batch"]), probs[None, :, None, :], True)
    return prompts, decode


def prepare(case, seed):
    c = case
    prompts, decode = _inputs(c, seed)
    lens, probs = _lengths(c), _append_prob(c)
    H, Hq, D, B, L = c["kv_heads"], c["q_heads"], c["head_dim"], c["batch"], c["layers"]
    longest = max(lens) + c["steps"] + 1
    pages = sum(-(-_slot_bound(n + c["steps"] + 1, p) // _PAGE) + 1 for row in probs for p in row for n in lens)
    cache = DmcCache(L, B, Hq, H, D, _dtype(c), longest, pages, max(p[1].shape[0] for p in prompts[0]),
                     window=c["window"])
    s = {"case": c, "cache": cache, "prompts": prompts, "decode": decode}
    if c["kind"] == "generate":
        s["out"] = torch.empty_like(decode[0])
        if c["mode"] == "graph":
            # a step's inputs in one buffer (q, k, v of every layer), its outputs in another
            sizes = [x[0].numel() for x in decode]
            s["steps_flat"] = [torch.cat([x[i].reshape(-1) for x in decode]) for i in range(c["steps"])]
            flat = torch.empty(sum(sizes), dtype=_dtype(c), device="cuda")
            q, k, v = (t.view(x.shape[1:]) for t, x in zip(flat.split(sizes), decode))
            out = torch.empty_like(q)
            cache.reset()
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                for layer in range(L):
                    cache.decode(layer, q[layer], k[layer], v[layer], out[layer])
            s["flat"], s["step_out"], s["graph"] = flat, out, graph
    elif c["kind"] == "compress":
        s["heads"] = torch.arange(B * H, dtype=torch.int32, device="cuda")
        s["cap"] = _export_cap(c)
    else:
        s["out"] = [torch.empty_like(p[0]) for p in prompts[0]]
    return s


def run(state):
    c, cache = state["case"], state["cache"]
    cache.reset()
    if c["kind"] == "attend":
        for (q, k, v, cu, longest), out in zip(state["prompts"][0], state["out"]):
            cache.prefill_attention(0, q, k, v, cu, longest, out)
        return [state["out"], cache.lengths(0)]
    for layer, parts in enumerate(state["prompts"]):
        for q0, k, v, cu, longest in parts:
            cache.prefill(layer, q0, k, v, cu, longest)
    if c["kind"] == "compress":
        return list(cache.export_heads(0, state["heads"], state["cap"]))
    (q, k, v), out = state["decode"], state["out"]
    for i in range(c["steps"]):
        if c["mode"] == "layers":
            cache.decode_layers(0, q[i], k[i], v[i], out[i])
        elif c["mode"] == "graph":
            state["flat"].copy_(state["steps_flat"][i])
            state["graph"].replay()
            out[i].copy_(state["step_out"])
        else:
            for layer in range(c["layers"]):
                cache.decode(layer, q[i, layer], k[i, layer], v[i, layer], out[i, layer])
    return [out, [cache.lengths(layer) for layer in range(c["layers"])]]


# ---------------------------------------------------------------- the same in 64 bits, by plain torch

def _states(q0, k, v, window):
    """Of one sequence's tokens: each token's slot index [T, H], whether it is its segment's last token, and
    the state of its slot after it (k, v [T, H, D], z [T, H]): the omega-weighted mean of its segment so far
    (of the segment's last `window` tokens if window > 0)."""
    T, H, D = k.shape
    w = torch.sigmoid(q0.double().view(T, H, -1).mean(2))
    opens = k[..., 0] < 0
    opens[0] = True
    kd = k.double()
    kd[..., 0] = 0.0
    at = torch.arange(T, device=k.device)[:, None].expand(T, H)
    first = torch.where(opens, at, 0).cummax(0).values
    if window:
        first = torch.maximum(first, at - (window - 1))

    def span(x):  # sums of x[first .. t]
        acc = torch.cat([torch.zeros_like(x[:1]), x.cumsum(0)])
        idx = first if x.dim() == 2 else first[..., None].expand(T, H, x.shape[2])
        return acc[1:] - acc.gather(0, idx)

    z = span(w)
    sk = span(w[..., None] * kd) / z[..., None]
    sv = span(w[..., None] * v.double()) / z[..., None]
    last = torch.cat([opens[1:], torch.ones_like(opens[:1])])
    return opens.long().cumsum(0) - 1, last, sk, sv, z


def _slots(slot, last, x, n):
    """The segments' final states as [H, n, ...]."""
    out = torch.zeros((slot.shape[1], n) + x.shape[2:], dtype=torch.float64, device=x.device)
    t, h = last.nonzero(as_tuple=True)
    out[h, slot[t, h]] = x[t, h]
    return out


def _attention(q, slot, last, sk, sv, t0):
    """Outputs of the tokens t0.. (queries q [T - t0, Hq, D]): each sees the final states of the slots before
    its own, and its own slot as it is after it."""
    T, H, D = sk.shape
    G = q.shape[1] // H
    n = int(slot.max()) + 1
    fk, fv = _slots(slot, last, sk, n), _slots(slot, last, sv, n)
    out = torch.empty(q.shape, dtype=torch.float64, device=q.device)
    step = max(1, int(2e8 // (H * G * n)))
    for a in range(t0, T, step):
        b = min(T, a + step)
        m = max(1, int(slot[b - 1].max()))
        qd = q[a - t0:b - t0].double()
        qd[..., 0] = 0.0
        qd = qd.view(b - a, H, G, D).permute(1, 0, 2, 3)                            # [H, t, G, D]
        dk, dv = sk[a:b].permute(1, 0, 2)[:, :, None], sv[a:b].permute(1, 0, 2)[:, :, None]
        s = (qd.reshape(H, -1, D) @ fk[:, :m].transpose(1, 2)).view(H, b - a, G, m)
        seen = torch.arange(m, device=q.device) < slot[a:b].t()[:, :, None, None]
        s = s.masked_fill(~seen, -math.inf)
        s = torch.cat([s, (qd * dk).sum(3, keepdim=True)], 3) / math.sqrt(D)
        p = torch.softmax(s, 3)
        o = (p[..., :m].reshape(H, -1, m) @ fv[:, :m]).view(H, b - a, G, D) + p[..., m:] * dv
        out[a - t0:b - t0] = o.permute(1, 0, 2, 3).reshape(b - a, H * G, D)
    return out


def exact(case, seed):
    c = case
    prompts, decode = _inputs(c, seed)
    lens, H, D = _lengths(c), c["kv_heads"], c["head_dim"]

    def sequence(layer, s, which):  # one sequence's prompt q, k or v
        parts = prompts[layer]
        return torch.cat([p[which][int(p[3][s]):int(p[3][s + 1])] for p in parts])

    if c["kind"] == "attend":
        outs = [torch.empty(p[0].shape, dtype=torch.float64, device="cuda") for p in prompts[0]]
        for s, n in enumerate(lens):
            q = sequence(0, s, 0)
            slot, last, sk, sv, _ = _states(q[..., 0], sequence(0, s, 1), sequence(0, s, 2), 0)
            o = _attention(q, slot, last, sk, sv, 0)
            for i, p in enumerate(prompts[0]):
                a, b = _part(n, c["parts"], i)
                outs[i][int(p[3][s]):int(p[3][s + 1])] = o[a:b]
        return [outs, None]
    if c["kind"] == "compress":
        cap, NH = _export_cap(c), c["batch"] * H
        k, v = (torch.zeros(NH, cap, D, dtype=torch.float64, device="cuda") for _ in range(2))
        z = torch.zeros(NH, cap, dtype=torch.float64, device="cuda")
        for s in range(c["batch"]):
            slot, last, sk, sv, sz = _states(*(sequence(0, s, i) for i in range(3)), c["window"])
            for x, to in ((sk, k), (sv, v), (sz, z)):
                to[s * H:(s + 1) * H] = _slots(slot, last, x, cap)
        return [k, v, z, None]
    q, kd, vd = decode
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    for layer in range(c["layers"]):
        for s, n in enumerate(lens):
            q0 = torch.cat([sequence(layer, s, 0), q[:, layer, s, :, 0]])
            k = torch.cat([sequence(layer, s, 1), kd[:, layer, s]])
            v = torch.cat([sequence(layer, s, 2), vd[:, layer, s]])
            slot, last, sk, sv, _ = _states(q0, k, v, c["window"])
            out[:, layer, s] = _attention(q[:, layer, s], slot, last, sk, sv, n)
    return [out, [None] * c["layers"]]
