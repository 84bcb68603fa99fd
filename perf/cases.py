"""The work that users of this framework have it do, as timed cases: quantising a prompt's keys and values into a
packed cache, decoding against it (one query token, several, several sequences, from device or from host buffers),
and whole requests (prompt, then generated tokens).

Sizes are the ones of the benchmark configurations (1, 32 and 4 x 8 KV heads, 4096 to 131072 tokens, 2 to 4 bits,
groups of 32, 64 and 128), of the latency study's decoder layer (32 query heads, 8 KV heads, sink 32, recent 96) and
ragged ones between them.  A case is a dict of plain values; `kind` says which calls a pass makes:

  prefill   one innerq_quantize_prefill of a prompt; the result is the packed cache
  decode    one innerq_decode_attention over a filled cache (what every layer of a model pays per token)
  generate  a request: prefill, then `steps` times innerq_append_token + innerq_decode_attention
  host      the same from pinned host buffers with innerq_decode_step_host, each result waited for before the next step
  verify    one innerq_decode_attention_multi of `n_q` query tokens (verification of speculated tokens)
  serve     `seqs` sequences of different lengths on one page pool: a prefill each, then `steps` batched steps
"""
import math

import torch

from paper_2602_23200_b200 import binding as B

D = 128
INNER, OUTER, FP16 = B.GROUPING_INNER, B.GROUPING_OUTER, B.GROUPING_FP16
SYM, ASYM, HYBRID = B.MODE_SYM, B.MODE_ASYM, B.MODE_HYBRID
PAGE_TOKENS = 512

BASE = dict(kind="decode", batch=1, n_q_heads=32, n_kv_heads=8, n_tokens=4096, group=32, k_bits=2, v_bits=2, k_mode=HYBRID,
            v_mode=HYBRID, w_sink=4, w_recent=128, grouping=INNER, steps=0, n_q=1, seqs=1, data="normal")


def _case(name, **kw):
    c = dict(BASE, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    layer = dict(n_q_heads=32, n_kv_heads=8, w_sink=32, w_recent=96, group=32, data="heavy")
    mha = dict(n_q_heads=32, n_kv_heads=32, group=32)
    batch16 = dict(batch=16, n_q_heads=32, n_kv_heads=8, group=64, data="heavy")
    long4 = dict(batch=4, n_q_heads=32, n_kv_heads=8, group=128, w_recent=256)
    return [
        # the smallest call: one head, where launch and latency are all there is
        _case("decode_1head_4k_2bit", n_q_heads=1, n_kv_heads=1, n_tokens=4096),
        # one layer of an 8B-class model takes a short prompt (first-token latency of a chat turn)
        _case("prefill_layer_512_k3v3", kind="prefill", n_tokens=512, k_bits=3, v_bits=3, k_mode=SYM, v_mode=SYM, **layer),
        # a short chat request on the same layer: prompt of odd length, 64 generated tokens, mixed code widths
        _case("generate_layer_1001_k3v2", kind="generate", n_tokens=1001, steps=64, k_bits=3, v_bits=2, k_mode=SYM, **layer),
        # steady-state decode of a multi-head model at its full context
        _case("decode_mha32_32k_2bit", n_tokens=32768, **mha),
        # a document summarised: long ragged prompt, then a run of generated tokens
        _case("generate_mha32_30011_2bit", kind="generate", n_tokens=30011, steps=48, **mha),
        # a caller whose model lives on the host side of the bus: step by step from pinned buffers
        _case("host_mha32_8k_2bit", kind="host", n_tokens=8192, steps=32, **mha),
        # a batch of requests at the accurate setting
        _case("generate_b16_8k_4bit", kind="generate", n_tokens=8192, steps=32, k_bits=4, v_bits=4, **batch16),
        # long-context decode and its prompt
        _case("decode_b4_128k_2bit", n_tokens=131072, **long4),
        _case("prefill_b4_128k_2bit", kind="prefill", n_tokens=131072, **long4),
        # speculative decoding: five tokens verified in one call
        _case("verify_layer_16k_4bit", kind="verify", n_tokens=16384, n_q=5, k_bits=4, v_bits=4, **layer),
        # continuous batching: sixteen requests of 1 to 8 thousand tokens on a page pool
        _case("serve_16seqs_8k_2bit", kind="serve", n_tokens=8192, seqs=16, steps=16, n_q_heads=32, n_kv_heads=8, group=64, data="heavy"),
        # the outer-grouped cache that the method is compared with
        _case("decode_outer_b16_8k_4bit", n_tokens=8192, k_bits=4, v_bits=4, k_mode=ASYM, v_mode=ASYM, grouping=OUTER, **batch16),
    ]


def draw(rng):
    kind = rng.choice(["prefill", "prefill", "decode", "decode", "decode", "generate", "generate", "host", "verify", "serve"])
    hkv, r = rng.choice([1, 2, 4, 8, 8, 16, 32]), rng.choice([1, 1, 2, 4, 4, 8])
    if hkv * r > 64:
        r = 1
    batch = rng.choice([1, 1, 1, 2, 3, 4, 8, 16])
    most = {"prefill": 131072, "decode": 131072, "generate": 32768, "host": 32768, "verify": 65536, "serve": 8192}[kind]
    n = int(math.exp(rng.uniform(math.log(200), math.log(most))))
    while batch * hkv * n > 1 << 21 and batch > 1:       # half of the largest listed case
        batch //= 2
    n = min(n, (1 << 21) // (batch * hkv))
    if rng.random() < 0.4:                               # model code pads prompts to multiples of its block size
        n = max(256, n // 256 * 256)
    w_sink, w_recent = rng.choice([(4, 128), (4, 128), (32, 96), (4, 256)])
    grouping = rng.choice([INNER] * 8 + [OUTER] + ([FP16] if kind in ("decode", "generate") else [INNER]))
    k_bits, v_bits = rng.choice([(2, 2), (2, 2), (3, 3), (4, 4), (4, 4), (3, 2), (4, 2), (4, 3)])
    k_mode, v_mode = rng.choice([(HYBRID, HYBRID), (HYBRID, HYBRID), (ASYM, ASYM), (SYM, SYM), (SYM, HYBRID)])
    if grouping == OUTER:
        k_bits = v_bits = rng.choice([2, 4])
        k_mode = v_mode = ASYM
    c = _case(None, kind=kind, batch=batch, n_q_heads=hkv * r, n_kv_heads=hkv, n_tokens=n, group=rng.choice([32, 64, 128]),
              k_bits=k_bits, v_bits=v_bits, k_mode=k_mode, v_mode=v_mode, w_sink=w_sink, w_recent=w_recent, grouping=grouping,
              data=rng.choice(["normal", "heavy"]))
    if kind in ("generate", "host"):
        c["steps"] = rng.randint(8, 64)
    elif kind == "serve":
        c.update(batch=1, seqs=rng.randint(3, 24), steps=rng.randint(4, 24))
        while c["seqs"] * hkv * n > 1 << 21:
            c["seqs"] = max(2, c["seqs"] // 2)
            n = c["n_tokens"] = min(n, (1 << 20) // (2 * hkv))
    elif kind == "verify":
        c["n_q"] = rng.randint(2, 8)
    return c


# ---------------------------------------------------------------- inputs
def _lengths(c):
    """Tokens of every sequence of a case (all different in `serve`, from an eighth of the longest up)."""
    if c["kind"] != "serve":
        return [c["n_tokens"]]
    n, s = c["n_tokens"], c["seqs"]
    return [max(1, n - (7 * n * i) // (8 * max(1, s - 1)) - (13 * i) % 29) for i in range(s)]


class _Draw:
    """fp16 keys, values and queries: N(0, 1) with outlier key channels, or heavy tails (Student t values, log-normal
    key channels), as in the benchmark's synthetic workloads."""

    def __init__(self, c, seed):
        self.c, self.g = c, torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        h = c["n_kv_heads"]
        if c["data"] == "heavy":
            self.scale = torch.exp(self.normal(h, D)).clamp_(0.05, 50.0)
        else:
            self.scale = torch.ones(h, D, device="cuda")
            chan = torch.rand(h, D, generator=self.g, device="cuda").argsort(1)[:, :3]
            self.scale.scatter_(1, chan, 10.0 + 20.0 * torch.rand(h, 3, generator=self.g, device="cuda"))

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device="cuda")

    def keys(self, batch, *rest):
        """fp16 [batch, n_kv_heads, ..., D]"""
        h = self.c["n_kv_heads"]
        out = torch.empty(batch, h, *rest, D, dtype=torch.float16, device="cuda")
        for b in range(batch):
            out[b] = (self.normal(h, *rest, D) * self.scale.view(h, *([1] * len(rest)), D)).clamp_(-65504, 65504)
        return out

    def values(self, batch, *rest):
        h = self.c["n_kv_heads"]
        out = torch.empty(batch, h, *rest, D, dtype=torch.float16, device="cuda")
        for b in range(batch):
            x = self.normal(h, *rest, D)
            if self.c["data"] == "heavy":
                chi = torch.zeros_like(x)
                for _ in range(4):
                    chi += self.normal(h, *rest, D).square_()
                x = x / (chi / 4).sqrt_()
            out[b] = x.clamp_(-65504, 65504)
        return out

    def queries(self, *shape):
        return self.normal(*shape, D).half()


def _inputs(c, seed):
    """Prompts [(K, V)] of every sequence and the tensors of the steps."""
    d, b, hq, s = _Draw(c, seed), c["batch"], c["n_q_heads"], c["steps"]
    prompts = [(d.keys(b, n), d.values(b, n)) for n in _lengths(c)]
    x = {"prompts": prompts}
    if c["kind"] in ("generate", "host"):
        x["k"] = d.keys(b, s).transpose(1, 2).transpose(0, 1).contiguous()         # [steps, batch, n_kv_heads, D]
        x["v"] = d.values(b, s).transpose(1, 2).transpose(0, 1).contiguous()
        x["q"] = d.queries(s, b, hq)
    elif c["kind"] == "serve":                                                     # [steps, seqs, batch, heads, D]
        x["k"] = d.keys(c["seqs"], s).permute(2, 0, 1, 3).unsqueeze(2).contiguous()
        x["v"] = d.values(c["seqs"], s).permute(2, 0, 1, 3).unsqueeze(2).contiguous()
        x["q"] = d.queries(s, c["seqs"], 1, hq)
    elif c["kind"] == "verify":
        x["q"] = d.queries(b, c["n_q"], hq)
    else:
        x["q"] = d.queries(b, hq)
    return x


def _config(c):
    keys = ("batch", "n_q_heads", "n_kv_heads", "group", "k_bits", "v_bits", "k_mode", "v_mode", "w_sink", "w_recent", "grouping")
    return B.make_config(max_tokens=max(_lengths(c)) + c["steps"], k_normalize=1 if c["grouping"] == INNER else 0,
                         **{k: c[k] for k in keys})


def prepare(case, seed):
    c, x, cfg = case, _inputs(case, seed), _config(case)
    s = dict(x, kind=c["kind"], steps=c["steps"])
    if c["kind"] == "serve":
        per_seq = [-(-(n + c["steps"]) // PAGE_TOKENS) for n in _lengths(c)]
        pool = B.PagePool(cfg, PAGE_TOKENS, sum(per_seq))
        pool.buf.zero_()
        s["pool"], s["caches"] = pool, [B.InnerQCache(cfg, pool=pool) for _ in per_seq]
        for cache, n in zip(s["caches"], _lengths(c)):
            cache.ensure_pages(n + c["steps"])
    else:
        s["caches"] = [B.InnerQCache(cfg)]
    if c["kind"] in ("decode", "verify"):
        s["caches"][0].innerq_quantize_prefill(*x["prompts"][0])
        del s["prompts"], x["prompts"]
    if c["kind"] == "host":
        for k in ("k", "v", "q"):
            s[k] = s[k].cpu().pin_memory()
    if c["kind"] in ("generate", "host", "serve"):
        s["out"] = torch.empty(s["q"].shape, dtype=torch.float16, pin_memory=True) if c["kind"] == "host" else torch.empty_like(s["q"])
        s["tokens"] = list(zip(s["k"], s["v"], s["q"], s["out"]))
    return s


def run(state):
    s, cache, kind = state, state["caches"][0], state["kind"]
    if kind == "prefill":
        cache.innerq_quantize_prefill(*s["prompts"][0])
        return {"cache": cache._cache_buf}                # the caller's own device buffer, which holds the packed cache
    if kind == "decode":
        return {"out": cache.innerq_decode_attention(s["q"])}
    if kind == "verify":
        return {"out": cache.innerq_decode_attention_multi(s["q"])}
    if kind == "serve":
        for ch, (k, v) in zip(s["caches"], s["prompts"]):
            ch.innerq_quantize_prefill(k, v)
        for k, v, q, out in s["tokens"]:
            B.innerq_append_token_batched(s["caches"], k, v)
            B.innerq_decode_attention_batched(s["caches"], q, out)
        return {"out": s["out"], "pages": s["pool"].buf}
    cache.innerq_quantize_prefill(*s["prompts"][0])
    if kind == "host":
        stream = torch.cuda.current_stream()
        for k, v, q, out in s["tokens"]:
            cache.innerq_decode_step_host(k, v, q, out)
            stream.synchronize()                          # the host reads this step's result before it makes the next
    else:
        for k, v, q, out in s["tokens"]:
            cache.innerq_append_token(k, v)
            cache.innerq_decode_attention(q, out)
    return {"out": s["out"], "cache": cache._cache_buf}


# ---------------------------------------------------------------- what a pass cannot do without
def _counts(c, n):
    """(packed key tokens, packed value tokens) of n cached tokens."""
    if c["grouping"] == FP16:
        return 0, 0
    row = max(0, n - c["w_sink"] - c["w_recent"])
    blk = row // c["group"] * c["group"]
    return (row, blk) if c["grouping"] == INNER else (blk, row)


def _cache_bytes(c, n):
    """Bytes that one unit's n cached tokens take: codes, scale (and zero-point) words, fp16 windows."""
    total = 0.0
    for nq, bits, mode in zip(_counts(c, n), (c["k_bits"], c["v_bits"]), (c["k_mode"], c["v_mode"])):
        total += nq * (16 * bits + (2 if mode == SYM else 4) * D / c["group"]) + (n - nq) * 2 * D
    return total


def work(case):
    c, units, hq = case, case["batch"] * case["n_kv_heads"], case["batch"] * case["n_q_heads"]
    total = flops = 0.0
    for n in _lengths(c):
        if c["kind"] not in ("decode", "verify"):         # prompt read, packed cache written
            total += units * (n * 4 * D + _cache_bytes(c, n))
            flops += units * n * D * 20.0
        steps = {"prefill": 0, "decode": 1, "verify": 1}.get(c["kind"], c["steps"])
        for t in range(steps):
            m = n if c["kind"] in ("decode", "verify") else n + t + 1
            total += units * (_cache_bytes(c, m) + 4 * D) + hq * c["n_q"] * 4 * D + (0 if m == n else units * 8 * D)
            flops += 4.0 * hq * c["n_q"] * m * D
    return {"bytes": total, "flops": flops}


def tolerance(case):
    # Outputs are fp16 (relative rounding error 2^-12 on average) of sums whose weights carry 16 bits and whose queries
    # carry 15; packed bytes have to be the same.
    return {"rel": 2e-3, "max": 2e-2}


# ---------------------------------------------------------------- the same in 64 bits
def _quantised(x, bits, mode, grp):
    """float64 values that a decoder sees for groups along the last axis of x (float32): the stored scale and zero-point
    are fp16 and codes come from them in correctly rounded float32 steps, which is part of the format."""
    top = 2 ** bits - 1
    g = x.reshape(*x.shape[:-1], -1, grp)
    mn, mx = g.amin(-1, keepdim=True), g.amax(-1, keepdim=True)
    s_a, z = ((mx - mn) / top).half().float(), mn.half().float()
    u = torch.where(s_a == 0, 0.0, torch.clamp(torch.round((g - z) * (1.0 / s_a)), 0, top))
    y_a = s_a.double() * u.double() + z.double()
    den = 2 ** (bits - 1) - 1
    s_s = (torch.maximum(mn.abs(), mx.abs()) / den).half().float()
    u = torch.where(s_s == 0, 0.0, torch.clamp(torch.round(g * (1.0 / s_s)), -den, den))
    y_s = s_s.double() * u.double()
    if mode == SYM:
        y = y_s
    elif mode == ASYM:
        y = y_a
    else:
        e_a, e_s = ((g.double() - y).abs().sum(-1, keepdim=True) for y in (y_a, y_s))
        y = torch.where(e_a < e_s, y_a, y_s)
    return y.reshape(x.shape)


def _attend(c, k, v, n_prompt, q, cached, visible):
    """One unit.  k, v: fp16 [T, D], prompt and later tokens; q: fp16 [S, r, D]; the cache holds cached[i] tokens at
    query i, which sees the first visible[i].  -> float64 [S, r, D]"""
    T, S, r = k.shape[0], q.shape[0], q.shape[1]
    kd, vd = k.double(), v.double()
    Q = q.double().reshape(S * r, D) / math.sqrt(D)
    pos = torch.arange(T, device=k.device)[:, None]
    scores = kd @ Q.T
    n_k, n_v = zip(*[_counts(c, m) for m in cached])
    k_packed = v_packed = torch.zeros(T, S, dtype=torch.bool, device=k.device)
    y_v = vd
    if c["grouping"] != FP16 and max(n_k + n_v) > 0:
        s0, G = c["w_sink"], c["group"]

        def tokens(x, n, bits, mode, rows):
            z = x.double()
            if n > 0:
                m = x[s0:s0 + n].float()
                z[s0:s0 + n] = _quantised(m, bits, mode, G) if rows else _quantised(m.T.contiguous(), bits, mode, G).T
            return z

        inner = c["grouping"] == INNER
        norm = torch.ones(D, device=k.device)
        if inner:
            norm = k[:n_prompt].float().abs().amax(0).sqrt()
            norm = torch.where(norm == 0, 1.0, norm)
        k_in = k.float()
        k_in[s0:] *= 1.0 / norm
        y_k = tokens(k_in, max(n_k), c["k_bits"], c["k_mode"], inner) * norm.double()
        y_v = tokens(v, max(n_v), c["v_bits"], c["v_mode"], not inner)
        lim = torch.tensor([n_k, n_v], device=k.device) + s0
        k_packed, v_packed = (pos >= s0) & (pos < lim[0]), (pos >= s0) & (pos < lim[1])
        scores = torch.where(k_packed.repeat_interleave(r, 1), y_k @ Q.T, scores)
    seen = pos < torch.tensor(visible, device=k.device)
    p = torch.softmax(scores.masked_fill(~seen.repeat_interleave(r, 1), -math.inf), 0)
    v_packed = v_packed.repeat_interleave(r, 1)
    out = (p * v_packed).T @ y_v + (p * ~v_packed).T @ vd
    return out.reshape(S, r, D)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "prefill":
        return None                                       # packed bytes only: compared as they are
    x, hkv, r = _inputs(c, seed), c["n_kv_heads"], c["n_q_heads"] // c["n_kv_heads"]
    per_seq = []
    for i, (k, v) in enumerate(x["prompts"]):
        n, s = k.shape[2], c["steps"]
        if kind == "verify":
            q, cached, visible = x["q"].transpose(0, 1), [n] * c["n_q"], [n - c["n_q"] + 1 + t for t in range(c["n_q"])]
        elif kind == "decode":
            q, cached, visible = x["q"][None], [n], [n]
        else:
            q = x["q"][:, i] if kind == "serve" else x["q"]
            kn, vn = (x["k"][:, i], x["v"][:, i]) if kind == "serve" else (x["k"], x["v"])
            cached = visible = [n + t + 1 for t in range(s)]
        out = torch.empty(q.shape, dtype=torch.float64, device="cuda")                    # [S, batch, n_q_heads, D]
        for b in range(c["batch"]):
            for h in range(hkv):
                ku, vu = k[b, h], v[b, h]
                if kind in ("generate", "host", "serve"):
                    ku, vu = torch.cat([ku, kn[:, b, h]]), torch.cat([vu, vn[:, b, h]])
                out[:, b, h * r:(h + 1) * r] = _attend(c, ku, vu, n, q[:, b, h * r:(h + 1) * r], cached, visible)
        per_seq.append(out)
    out = per_seq[0]
    if kind == "serve":
        return {"out": torch.stack(per_seq, 1), "pages": None}
    if kind == "verify":
        return {"out": out.transpose(0, 1).contiguous()}
    if kind == "decode":
        return {"out": out[0]}
    return {"out": out, "cache": None}
