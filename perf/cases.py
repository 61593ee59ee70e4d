"""The measured cases: the calls that a program using this library makes, with
inputs, output tolerances and the work none of them can do without.

Five kinds of case, all through the public binding:

  linear    ssd_linear_noalloc: one projection on the caller's device tensors
  forward   ssd_debug_forward: one decoder forward that returns its logits -
            a decode step (1 row), a draft step (1 row, half of the sublayers
            skipped) or a verification (K + 1 rows) over a filled KV cache
  prefill   ssd_prefill of a prompt, then the forward of its last token: the
            time until the first logits are there
  generate  ssd_generate (prompt encoding, K drafts and a verification per
            round), then the logits of the next position over the whole
            cache it left, so that more than token ids is compared
  sample    the same in sampling mode (temperature 1, top-p 0.95)

Forward and prefill cases run models of 2 to 4 layers at the widths of the
workloads (bf16 weights far larger than L2); one generate case is the 7B shape
at its full depth.

Weights are Gaussian with a scale of 1 / sqrt(fan-in) (0.02 at d = 4096) and
norm gains near 1; the output projections are divided by sqrt(2 L), and those
of skipped sublayers scaled by 0.05.  As in a trained model, and unlike random
initialisation, the next token is mostly predictable: every token has four
likely successors (lm_head rows hold multiples of their predecessors'
embeddings), so that drafts are usually accepted and a token does not hang on
the last bit of a sum.
"""
import math

import numpy as np
import torch

import paper_2309_08168_gb300 as ssd

_TINY = dict(layers=4, d=256, heads=4, kv_heads=4, hd=64, ffn=688, vocab=2048)
_7B = dict(layers=4, d=4096, heads=32, kv_heads=32, hd=128, ffn=11008, vocab=32000)
_13B = dict(layers=4, d=5120, heads=40, kv_heads=40, hd=128, ffn=13824, vocab=32000)
_70B = dict(layers=2, d=8192, heads=64, kv_heads=8, hd=128, ffn=28672, vocab=32000)


def listed():
    return [
        # smallest call: a ragged projection, latency and launches only
        dict(name="linear_small", kind="linear", M=1, K=528, N=100),
        # a square projection for a full batch of verification rows
        dict(name="linear_square", kind="linear", M=16, K=4096, N=4096),
        # a vocabulary head, the largest output that the fixed scratch allows
        dict(name="linear_head", kind="linear", M=4, K=4096, N=32000),
        # the smallest whole generation: a short prompt, 64 tokens, launches and barriers
        dict(name="generate_tiny", kind="generate", **_TINY, prompt=32, n_new=64, rows=5),
        # plain autoregressive step in mid-generation, odd context
        dict(name="decode_7b", kind="forward", **_7B, ctx=701, rows=1, draft=False),
        # drafting step with grouped-query attention, the bulk of a 70B round
        dict(name="draft_70b", kind="forward", **dict(_70B, layers=4), ctx=1151, rows=1, draft=True),
        # verification of 8 drafts
        dict(name="verify_7b", kind="forward", **_7B, ctx=767, rows=9, draft=False),
        # verification of 12 drafts near the end of the longest cache
        dict(name="verify_13b", kind="forward", **_13B, ctx=2035, rows=13, draft=False),
        # prompt encoding, ordinary and large
        dict(name="prefill_7b", kind="prefill", **_7B, prompt=512, rows=1),
        dict(name="prefill_70b", kind="prefill", **_70B, prompt=1024, rows=1),
        # a whole greedy call at full depth: prompt, drafting, verification, acceptance
        dict(name="generate_7b", kind="generate", **dict(_7B, layers=32), prompt=512, n_new=64, rows=9),
        # a whole sampling call with a long prompt
        dict(name="sample_13b", kind="sample", **dict(_13B, layers=6), prompt=1536, n_new=26, rows=13),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["linear", "linear", "forward", "forward", "forward", "prefill", "prefill", "generate", "sample"])
    if kind == "linear":
        while True:
            M, K, N = rng.randint(1, 16), 16 * _log(rng, 2, 512), _log(rng, 24, 32768)
            if K <= 512 or -(-K // 512) * M * 64 * -(-N // 64) <= 1 << 20:  # the call's fixed scratch
                return dict(kind=kind, M=M, K=K, N=N)
    hd = rng.choice([64, 128, 128])
    unit = 128 // hd  # heads per 128 features
    if kind in ("forward", "prefill"):
        d = 128 * _log(rng, 4, 64)
        layers = rng.randint(1, 4)
    else:
        d = 128 * _log(rng, 4, 40)
        layers = rng.randint(2, 8)
    kv = unit * max(1, d // 128 // rng.choice([1, 1, 2, 4, 8]))
    heads = kv * max(1, d // hd // kv)
    m = dict(kind=kind, layers=layers, d=d, heads=heads, kv_heads=kv, hd=hd, ffn=16 * int(d * rng.uniform(2.5, 3.5) / 16),
             vocab=_log(rng, 1000, 32768))
    if kind == "forward":
        draft = rng.random() < 0.4
        return dict(m, ctx=_log(rng, 20, 2100), rows=1 if draft else rng.randint(1, 16), draft=draft)
    if kind == "prefill":
        return dict(m, prompt=_log(rng, 20, 2300), rows=1)
    return dict(m, prompt=_log(rng, 20, 1600), n_new=rng.randint(8, 48) if kind == "generate" else rng.randint(8, 26),
                rows=rng.randint(1, 13))


# -- inputs -------------------------------------------------------------------

def _skip(c):
    """Half of the sublayers, the middle of the network."""
    return [1 if c["layers"] // 2 <= s < (3 * c["layers"]) // 2 else 0 for s in range(2 * c["layers"])]


def _weights(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    L, d, qd, kvd, F, V = c["layers"], c["d"], c["heads"] * c["hd"], c["kv_heads"] * c["hd"], c["ffn"], c["vocab"]
    skip = _skip(c)

    def mat(n, k, scale):
        return torch.empty(n, k, dtype=torch.bfloat16, device="cuda").normal_(0.0, scale / math.sqrt(k), generator=g)

    def gain():
        return torch.empty(d, dtype=torch.bfloat16, device="cuda").normal_(1.0, 0.1, generator=g)

    w = {"embed": mat(V, d, math.sqrt(d)), "final_norm": gain(), "layers": []}
    head = mat(V, d, 1.28).float()
    for level in (24.0, 22.5, 21.5, 19.5):  # four likely successors of every token
        head[torch.randperm(V, generator=g, device="cuda")] += w["embed"].float() * (level / d)
    w["lm_head"] = head.to(torch.bfloat16)
    for l in range(L):
        so = (0.05 if skip[2 * l] else 1.0) / math.sqrt(2 * L)
        sd = (0.05 if skip[2 * l + 1] else 1.0) / math.sqrt(2 * L)
        w["layers"].append({
            "wq": mat(qd, d, 1.28), "wk": mat(kvd, d, 1.28), "wv": mat(kvd, d, 1.28), "wo": mat(d, qd, 4.0 * so),
            "attn_norm": gain(), "w_gate": mat(F, d, 1.28), "w_up": mat(F, d, 1.28), "w_down": mat(d, F, 1.5 * sd),
            "mlp_norm": gain()})
    return w


def _tokens(c, seed, n):
    return np.random.default_rng(seed + 77).integers(0, c["vocab"], n, dtype=np.int32)


def _linear_inputs(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.empty(c["N"], c["K"], dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0 / math.sqrt(c["K"]), generator=g)
    x = torch.randn(c["M"], c["K"], device="cuda", generator=g)
    return w, x


def prepare(case, seed):
    if case["kind"] == "linear":
        w, x = _linear_inputs(case, seed)
        return {"case": case, "w": w, "x": x, "y": torch.empty(case["M"], case["N"], device="cuda")}
    w = _weights(case, seed)
    torch.cuda.synchronize()  # the decoder runs on a stream of its own
    if case["kind"] == "forward":
        n = case["ctx"] + case["rows"]
    else:
        n = case["prompt"] + case.get("n_new", 0) + case["rows"]
    cfg = ssd.make_config(case["layers"], case["d"], case["heads"], case["kv_heads"], case["hd"], case["ffn"],
                          case["vocab"], n + 1)
    dec = ssd.Decoder(cfg, w, on_device=True)
    dec.set_skip(_skip(case))
    dec.set_sampling(1.0, 0.95)
    s = {"case": case, "dec": dec, "seed": seed}
    if case["kind"] == "forward":
        t = _tokens(case, seed, n)
        dec.prefill(t[: case["ctx"] + 1])  # fills the cache up to the position of the forward
        s["rows"] = t[case["ctx"]:]
    else:
        s["prompt"] = _tokens(case, seed, case["prompt"])
    return s


def run(state):
    c = state["case"]
    if c["kind"] == "linear":
        ssd.ssd_linear_noalloc(state["w"], state["x"], state["y"], c["N"], c["K"], c["M"],
                               torch.cuda.current_stream().cuda_stream)
        return state["y"]
    dec = state["dec"]
    if c["kind"] == "forward":
        return dec.debug_forward(c["draft"], state["rows"], c["ctx"])
    if c["kind"] == "prefill":
        dec.prefill(state["prompt"])
        return dec.debug_forward(False, state["prompt"][-1:], c["prompt"] - 1)
    mode = ssd.SSD_SAMPLE if c["kind"] == "sample" else ssd.SSD_GREEDY
    toks, _ = dec.generate(state["prompt"], c["n_new"], c["rows"] - 1, mode, state["seed"])
    return toks, dec.debug_forward(False, toks[-1:], c["prompt"] - 1 + c["n_new"])


# -- the work of one pass -------------------------------------------------------

def _forward_work(c, rows, ctx, draft, logits=True):
    """Weights and KV read once, one pass of multiply-adds per row (logits rows written)."""
    qd, kvd, d = c["heads"] * c["hd"], c["kv_heads"] * c["hd"], c["d"]
    skip = _skip(c) if draft else [0] * (2 * c["layers"])
    n_a, n_m = skip[0::2].count(0), skip[1::2].count(0)
    params = n_a * (2 * qd * d + 2 * kvd * d) + n_m * 3 * c["ffn"] * d
    head = c["vocab"] * d if logits else 0
    kv = n_a * 2 * kvd * (ctx + rows) * 2
    seen = ctx * rows + rows * (rows + 1) / 2
    return (2.0 * (params + head + rows * d) + kv + (4.0 * rows * c["vocab"] if logits else 0),
            2.0 * rows * (params + head) + n_a * 4.0 * qd * seen)


def work(case):
    c = case
    if c["kind"] == "linear":
        return {"bytes": 2.0 * c["N"] * c["K"] + 4.0 * c["M"] * (c["K"] + c["N"]), "flops": 2.0 * c["M"] * c["N"] * c["K"]}
    if c["kind"] == "forward":
        b, f = _forward_work(c, c["rows"], c["ctx"], c["draft"])
        return {"bytes": b, "flops": f}
    p = c["prompt"] - 1
    b, f = _forward_work(c, p, 0, False, logits=False)
    steps = [(1, p, False)]  # the forward after a prefill
    if c["kind"] != "prefill":
        # as many rounds as there are when every draft is accepted
        K, left, at, steps = c["rows"] - 1, c["n_new"], p, []
        while left > 0:
            k = min(K, left - 1)
            steps += [(1, at + j, True) for j in range(k)] + [(k + 1, at, False)]
            at, left = at + k + 1, left - k - 1
        steps.append((1, at, False))
    for rows, ctx, draft in steps:
        x, y = _forward_work(c, rows, ctx, draft)
        b, f = b + x, f + y
    return {"bytes": b, "flops": f}


def tolerance(case):
    if case["kind"] == "linear":
        # inputs enter as bf16 pairs (16 bits), 32-bit sums
        return {"rel": 1e-5, "max": 1e-4}
    # fp16 keys and values, inputs as bf16 pairs, 32-bit sums over all layers
    t = {"rel": 1.2e-3, "max": 1e-2}
    if case["kind"] in ("generate", "sample"):
        t["differ"] = 0.0
    return t


# -- the same in 64 bits ----------------------------------------------------------

def _rms(x, g):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-5) * g.double()


def _rope(x, pos, hd):
    f = pos.double()[:, None] * (1e4 ** (-torch.arange(0, hd, 2, device="cuda", dtype=torch.float64) / hd))[None]
    c, s = f.cos()[:, None], f.sin()[:, None]
    a, b = x[..., : hd // 2], x[..., hd // 2:]
    return torch.cat([a * c - b * s, b * c + a * s], -1)


def _attend(q, k, v, pos0, hd):
    """q [n][H][hd] at positions pos0.., k and v [t][Hkv][hd]; 256 rows at a time."""
    rep = q.shape[1] // k.shape[1]
    k, v = k.repeat_interleave(rep, 1).transpose(0, 1), v.repeat_interleave(rep, 1).transpose(0, 1)
    out = []
    for r in range(0, q.shape[0], 256):
        x = q[r: r + 256].transpose(0, 1) @ k.transpose(1, 2) / math.sqrt(hd)
        at = pos0 + r + torch.arange(x.shape[1], device="cuda")
        x.masked_fill_(torch.arange(k.shape[1], device="cuda")[None] > at[:, None], -math.inf)
        out.append((x.softmax(-1) @ v).transpose(0, 1))
    return torch.cat(out).reshape(q.shape[0], -1)


def _model(c, w, tokens, pos0, cache, skip, logits):
    """Rows `tokens` at positions pos0.. over the cache (a list of (K, V) by layer, replaced by the extended one)."""
    t = torch.as_tensor(np.asarray(tokens), device="cuda").long()
    pos = pos0 + torch.arange(t.numel(), device="cuda")
    h, hd = w["embed"][t].double(), c["hd"]
    for l, y in enumerate(w["layers"]):
        if not skip[2 * l]:
            x = _rms(h, y["attn_norm"])
            q = _rope((x @ y["wq"].double().T).view(-1, c["heads"], hd), pos, hd)
            k = _rope((x @ y["wk"].double().T).view(-1, c["kv_heads"], hd), pos, hd)
            v = (x @ y["wv"].double().T).view(-1, c["kv_heads"], hd)
            if cache[l] is not None:
                k, v = torch.cat([cache[l][0][:pos0], k]), torch.cat([cache[l][1][:pos0], v])
            cache[l] = (k, v)
            h = h + _attend(q, k, v, pos0, hd) @ y["wo"].double().T
        if not skip[2 * l + 1]:
            x = _rms(h, y["mlp_norm"])
            h = h + (torch.nn.functional.silu(x @ y["w_gate"].double().T) * (x @ y["w_up"].double().T)) @ y["w_down"].double().T
    return _rms(h, w["final_norm"]) @ w["lm_head"].double().T if logits else None


def exact(case, seed):
    c = case
    if c["kind"] == "linear":
        w, x = _linear_inputs(c, seed)
        return x.double() @ w.double().T
    if c["kind"] == "sample" or c.get("n_new", 0) * c["layers"] > 300:
        return None  # random choices; or too many steps for 64 bits
    w, none, cache = _weights(c, seed), [0] * (2 * c["layers"]), [None] * c["layers"]
    if c["kind"] == "forward":
        t = _tokens(c, seed, c["ctx"] + c["rows"])
        _model(c, w, t[: c["ctx"]], 0, cache, none, False)
        return _model(c, w, t[c["ctx"]:], c["ctx"], cache, _skip(c) if c["draft"] else none, True).cpu().numpy()
    t = _tokens(c, seed, c["prompt"])
    p = c["prompt"] - 1
    _model(c, w, t[:p], 0, cache, none, False)
    out = _model(c, w, t[p:], p, cache, none, True)
    if c["kind"] == "prefill":
        return out.cpu().numpy()
    toks = []
    for i in range(c["n_new"]):
        toks.append(int(out[0].argmax()))
        out = _model(c, w, toks[-1:], p + 1 + i, cache, none, True)
    return np.asarray(toks, dtype=np.int32), out.cpu().numpy()
