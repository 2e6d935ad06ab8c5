"""What the performance of this library is measured on: calls a user's program makes, over the range it makes them in.

Three kinds of work go through the public entry points of the package:
  generate  sdfp_generate (speculative or autoregressive decoding of a batch of prompts), then the logits of the last
            positions of the first sequence from sdfp_forward_logits, as a program that reports probabilities asks for them
  score     the logits of every position of a text, sdfp_forward_logits chunk by chunk
  fit       sdfp_fit_scores, the per-layer sensitivities from which the layers to prune are chosen
A case states the decoder's dimensions, how it is decoded and what it is fed.

Weights are random, but predict as a trained decoder does: with a clear favourite.  The embedding of token t pulls the
lm-head's row of t's successor; a layer the draft leaves out holds facts (for some tokens t an FFN unit that answers t and
moves the residual stream towards another token's successor), so the draft is wrong after exactly those tokens.  The
attention and FFN blocks around that are dense random matrices that carry half of the residual stream's energy.  Near-ties,
which rounding decides, do not occur except by rare accident, and the acceptance rate is that of a useful draft.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2602_05499_b200 as sdfp

HARD = 0.15      # share of tokens after which the draft is wrong
TAIL_ROWS = 8    # positions whose logits a generate case returns


def _case(kind, layers, heads, head_dim, ffn, vocab, dtype="bf16", **kw):
    c = dict(kind=kind, layers=layers, heads=heads, head_dim=head_dim, ffn=ffn, vocab=vocab, dtype=dtype)
    if kind == "generate":
        c.update(skip_attn=0, skip_ffn=0, share_kv=False, k=4, batch=1, prompt=512, new=64, temperature=0.0)
    c.update(kw)
    return c


def listed():
    tiny = dict(layers=4, heads=4, head_dim=64, ffn=688, vocab=2048)          # the test-size decoder of synth_inputs
    d4096 = dict(heads=32, head_dim=128, ffn=11008, vocab=32000)              # synth_inputs.LLAMA7B's layers
    d5120 = dict(heads=40, head_dim=128, ffn=13824, vocab=32000)              # synth_inputs.LLAMA13B's layers
    return [
        # the smallest call: a test-size fp32 decoder, speculative; a pass is all latency
        dict(_case("generate", **tiny, dtype="f32", skip_attn=2, skip_ffn=2, k=4, prompt=16, new=64), name="tiny-f32-greedy-k4"),
        # a small bf16 decoder without a draft: plain autoregressive decoding from a short prompt
        dict(_case("generate", **tiny, k=0, prompt=21, new=48), name="tiny-bf16-ar"),
        # the headline workload at full depth: one sequence, prompt of 512, greedy, k = 4, 12 of 32 layers pruned
        dict(_case("generate", 32, **d4096, skip_attn=12, skip_ffn=12, k=4, prompt=512, new=64), name="d4096-greedy-k4"),
        # the vanilla baseline of that workload, shallower, ragged prompt
        dict(_case("generate", 16, **d4096, k=0, prompt=201, new=32), name="d4096-ar"),
        # rejection sampling at temperature 1 with a longer draft
        dict(_case("generate", 16, **d4096, skip_attn=6, skip_ffn=6, k=6, prompt=333, new=48, temperature=1.0), name="d4096-sampled-k6"),
        # a long prompt on the wider layers: the prompt pass and the long cache
        dict(_case("generate", 10, **d5120, skip_attn=4, skip_ffn=4, k=4, prompt=2048, new=48), name="d5120-long-prompt"),
        # attention and FFN blocks pruned at different ratios, the draft in the target's cache
        dict(_case("generate", 10, **d5120, skip_attn=5, skip_ffn=3, share_kv=True, k=3, prompt=777, new=40), name="d5120-sublayer-shared-kv"),
        # a batch of eight sequences with long prompts
        dict(_case("generate", 16, **d4096, skip_attn=6, skip_ffn=6, k=4, batch=8, prompt=1024, new=32), name="d4096-batch8-k4"),
        # the widest batch with short prompts (chat turns), 48 rows per verify pass
        dict(_case("generate", 12, **d4096, skip_attn=4, skip_ffn=4, k=2, batch=16, prompt=45, new=24), name="d4096-batch16-short"),
        # scoring a short text position by position
        dict(_case("score", 8, **d4096, length=75), name="d4096-score"),
        # layer sensitivities of a few full-width layers
        dict(_case("fit", 4, **d4096, sequences=2, length=65), name="d4096-fit"),
        # layer sensitivities of the test-size fp32 decoder, eight sequences of 32 tokens
        dict(_case("fit", **tiny, dtype="f32", sequences=8, length=32), name="tiny-f32-fit"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: small fp32 and bf16 decoders, wide bf16 layers, one sequence and batches."""
    kind = rng.choice(["generate"] * 7 + ["score"] + ["fit"] * 2)
    small = rng.random() < 0.35
    dtype = "bf16" if not small or rng.random() < 0.4 else "f32"
    head_dim = 64 if small else rng.choice([64, 128, 128])
    heads = _log(rng, 256, 768) // 64 if small else _log(rng, 2048, 5120) // head_dim
    d = heads * head_dim
    ffn = 16 * int(d * rng.uniform(2.4, 3.2) / 16)
    vocab = 16 * (_log(rng, 1024, 8192) if small else _log(rng, 8192, 32000)) // 16 // 16 * 16
    layers = rng.randint(3, 6) if small else rng.randint(4, 10)
    if kind == "fit":
        layers = min(layers, 4)
        return _case(kind, layers, heads, head_dim, ffn, vocab, dtype, sequences=rng.randint(1, 8 if small else 3), length=rng.randint(17, 80))
    if kind == "score":
        return _case(kind, layers, heads, head_dim, ffn, vocab, dtype, length=_log(rng, 3, 160))
    k = rng.choice([0, 2, 3, 4, 4, 5, 6, 8])
    batch = rng.choice([1, 1, 1, 2, 3, 4, 6, 8, 12, 16])
    while batch * max(k + 1, 2) > 80:
        batch -= 1
    skip = 0 if k == 0 else rng.randint(1, max(1, layers // 2))
    skip_ffn = 0 if k == 0 else max(1, min(layers - 2, skip + rng.choice([-1, 0, 0, 0, 1])))
    prompt = _log(rng, 2, 256 if small else max(64, 2048 // batch))
    return _case(kind, layers, heads, head_dim, ffn, vocab, dtype, skip_attn=skip, skip_ffn=skip_ffn, share_kv=rng.random() < 0.25 and k > 0,
                 k=k, batch=batch, prompt=prompt, new=rng.randint(12, 48), temperature=rng.choice([0.0, 0.0, 0.0, 1.0]) if batch == 1 else 0.0)


def _keep(layers, n_skip):
    """1 = the draft runs the block: the n_skip layers in front of the last one are left out."""
    return np.array([0 if layers - 1 - n_skip <= l < layers - 1 else 1 for l in range(layers)], dtype=np.uint8)


def _weights(case, gen):
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    L, d, f, V = case["layers"], case["heads"] * case["head_dim"], case["ffn"], case["vocab"]

    def normal(rows, cols, std):
        return torch.randn(rows, cols, generator=gen, device="cuda", dtype=dt).mul_(std)

    embed = normal(V, d, 1.0)
    rho = min(0.8, 22.0 / math.sqrt(d))  # how strongly a token pulls its successor's row of the lm-head
    lm_head = normal(V, d, 0.02 * math.sqrt(1.0 - rho * rho))
    lm_head[torch.randperm(V, generator=gen, device="cuda")] += embed * (0.02 * rho)
    if case.get("temperature", 0.0) > 0.0:  # a second choice to sample, about a third as likely
        lm_head[torch.randperm(V, generator=gen, device="cuda")] += embed * (0.02 * rho * 0.95)
    one = torch.ones(d, device="cuda", dtype=dt)
    block = 1.0 / math.sqrt(2.0 * L)     # what a block adds to the residual stream, against the embedding's 1
    layers = []
    for _ in range(L):
        lw = {n: normal(d, d, 1.25 / math.sqrt(d)) for n in ("wq", "wk", "wv")}
        lw["wo"] = normal(d, d, 2.0 * block / math.sqrt(d))
        lw["w_gate"], lw["w_up"] = normal(f, d, 1.25 / math.sqrt(d)), normal(f, d, 1.25 / math.sqrt(d))
        lw["w_down"] = normal(d, f, 1.2 * block / math.sqrt(f))
        lw["attn_norm"], lw["ffn_norm"] = one, one
        layers.append(lw)
    if case.get("skip_ffn", 0) > 0:      # the facts of a pruned layer
        lw, n = layers[L - 2], min(int(HARD * V), f // 2)
        hard = torch.randperm(V, generator=gen, device="cuda")[:n]
        lw["w_gate"][:n] = embed[hard] * (8.0 / d)
        lw["w_up"][:n] = embed[hard] * (4.0 / d)
        lw["w_down"][:, :n] = embed[torch.randperm(V, generator=gen, device="cuda")[:n]].t() * (2.0 / 18.0)
    return {"tok_embed": embed, "lm_head": lm_head, "final_norm": one, "layers": layers}


def prepare(case, seed):
    """A decoder handed to the library (or, for fit, its weights) and the token ids of the call."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    rng = np.random.RandomState(int(seed) % (2**31 - 1))
    shape = SimpleNamespace(n_layers=case["layers"], d_model=case["heads"] * case["head_dim"], n_heads=case["heads"], head_dim=case["head_dim"],
                            d_ffn=case["ffn"], vocab=case["vocab"], rms_eps=1e-5, rope_theta=10000.0, dtype=case["dtype"])
    weights = _weights(case, gen)
    if case["kind"] == "fit":
        return dict(case=case, shape=shape, weights=weights, tokens=rng.randint(0, case["vocab"], (case["sequences"], case["length"])).astype(np.int32))
    if case["kind"] == "score":
        return dict(case=case, engine=sdfp.Sdfp(shape, weights, max_seq=case["length"] + 16), tokens=rng.randint(0, case["vocab"], case["length"]).astype(np.int32))
    engine = sdfp.Sdfp(shape, weights, max_seq=case["prompt"] + case["new"] + case["k"] + 8, max_batch=case["batch"], k_max=case["k"])
    if case["k"] > 0:
        engine.sdfp_set_draft_sublayers(_keep(case["layers"], case["skip_attn"]), _keep(case["layers"], case["skip_ffn"]))
        engine.sdfp_set_draft_kv_sharing(case["share_kv"])
    return dict(case=case, engine=engine, seed=int(seed), tokens=rng.randint(0, case["vocab"], (case["batch"], case["prompt"])).astype(np.int32))


def run(state):
    case, tokens = state["case"], state["tokens"]
    if case["kind"] == "fit":
        trace, fit = sdfp.sdfp_fit_scores(state["shape"], state["weights"], tokens)
        return {"trace": np.array(trace), "fit": np.array(fit)}
    engine = state["engine"]
    if case["kind"] == "score":
        return [engine.sdfp_forward_logits(tokens[i:i + 80], i) for i in range(0, len(tokens), 80)]
    out = engine.sdfp_generate(tokens, case["k"], case["new"], temperature=case["temperature"], seed=state["seed"])
    text = np.concatenate([tokens[0], np.asarray(out.tokens[0], dtype=np.int32)])
    rows = min(TAIL_ROWS, len(text))
    logits = engine.sdfp_forward_logits(text[-rows:], len(text) - rows)
    rounds = np.zeros((case["new"], case["batch"], 3), dtype=np.int32)  # drafted, accepted, committed; as many rows as there can be rounds
    rounds[:out.n_rounds] = out.stats
    return {"tokens": np.asarray(out.tokens), "rounds": rounds, "logits": logits}


def _sizes(case):
    d, f, e = case["heads"] * case["head_dim"], case["ffn"], 4 if case["dtype"] == "f32" else 2
    return d, 4 * d * d, 3 * d * f, case["vocab"] * d, e


def work(case):
    """Bytes and operations of one call.  Passes follow one another, so every pass reads its weights and its sequences'
    keys and values again, unless the whole model stays in the L2 cache."""
    d, attn, ffn, head, e = _sizes(case)
    L = case["layers"]
    body = L * (attn + ffn)
    if case["kind"] == "fit":  # a forward and a backward pass of all rows; the weights' mean squares ride along
        rows = case["sequences"] * (case["length"] - 1)
        return {"bytes": (2 * (body + head)) * e, "flops": 4 * rows * (body + head)}
    if case["kind"] == "score":
        return {"bytes": (body + head) * e * -(-case["length"] // 80) + 4 * case["length"] * case["vocab"], "flops": 2 * case["length"] * (body + head)}
    B, P, k, new = case["batch"], case["prompt"], case["k"], case["new"]
    per_round = (1 - (1 - HARD) ** (k + 1)) / HARD
    rounds = math.ceil(new / per_round) if k else new
    draft = ((L - case["skip_attn"]) * attn + (L - case["skip_ffn"]) * ffn + head) if k else 0
    decode = rounds * (k * draft + body + head)
    kv = 2 * d * e * (P + new / 2) * B  # keys and values of the batch, one layer, once
    weights = (body if P > 1 else 0) + decode + body + head  # the prompt, the rounds, the closing logits
    if (body + head) * e < 100e6:
        weights, kv = body + head, kv / max(1, rounds * (k + 1))
    cache = rounds * (k * (L - case["skip_attn"]) + L) * kv if k else rounds * L * kv
    rows = B * (P - 1)
    flops = 2 * rows * body + 2 * B * P * P * d * L + 2 * B * rounds * (k * draft + (k + 1) * (body + head))
    return {"bytes": weights * e + cache + 2 * d * e * L * rows, "flops": flops}


def tolerance(case):
    # Measured: the bf16 paths, which add in different orders, are up to 9e-4 (2-norm) and 5e-3 (largest) apart in the logits and
    # agree in every token; the sensitivities are within 1e-7 of the same sums in 64 bits; fp32 logits are sums of 32-bit values.
    if case["kind"] == "fit":
        return {"rel": 1e-5}
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.0} if case["dtype"] == "f32" else {"rel": 4e-3, "max": 2e-2, "differ": 0.0}


# ---- the same results in 64 bits ----
# Plain torch, one operation after another; the only rounding is the one the method states: keys and values of a bf16
# decoder are bf16 numbers in the cache.

def _norm(x, gain):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-5) * gain


def _rotate(x, pos):  # x [T, heads, head_dim]
    half = x.shape[-1] // 2
    angle = pos.double()[:, None] * (10000.0 ** (-torch.arange(half, device=x.device, dtype=torch.float64) / half))[None]
    c, s = torch.cos(angle).float().double()[:, None], torch.sin(angle).float().double()[:, None]  # tables of 32-bit numbers
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * c - b * s, b * c + a * s], -1)


class _Exact:
    def __init__(self, case, weights, grad=False):
        self.case, self.w, self.cache, self.grad = case, weights, [None] * case["layers"], grad

    def _attend(self, l, q, k, v):
        heads, hd = self.case["heads"], self.case["head_dim"]
        q, k, v = (t.view(len(t), heads, hd) for t in (q, k, v))
        before = 0 if self.cache[l] is None else len(self.cache[l][0])
        pos = torch.arange(before, before + len(q), device=q.device)
        q, k = _rotate(q, pos), _rotate(k, pos)
        if not self.grad:
            if self.case["dtype"] != "f32":
                k, v = k.bfloat16().double(), v.bfloat16().double()
            if before:
                k, v = torch.cat([self.cache[l][0], k]), torch.cat([self.cache[l][1], v])
            self.cache[l] = (k, v)
        see = torch.arange(len(k), device=q.device)[None] <= pos[:, None]
        out = [torch.softmax((q[:, h] @ k[:, h].t() / math.sqrt(hd)).masked_fill(~see, -math.inf), -1) @ v[:, h] for h in range(heads)]
        return torch.cat(out, -1)

    def logits(self, tokens, rows, layers=None):
        """Logits of the last `rows` of these tokens, which follow what the cache holds."""
        h = self.w["tok_embed"][torch.as_tensor(tokens, device="cuda").long()].double()
        for l in range(self.case["layers"]):
            lw = layers[l] if layers else {n: t.double() for n, t in self.w["layers"][l].items()}
            x = _norm(h, lw["attn_norm"])
            h = h + self._attend(l, x @ lw["wq"].t(), x @ lw["wk"].t(), x @ lw["wv"].t()) @ lw["wo"].t()
            x = _norm(h, lw["ffn_norm"])
            h = h + (torch.nn.functional.silu(x @ lw["w_gate"].t()) * (x @ lw["w_up"].t())) @ lw["w_down"].t()
        return _norm(h[len(h) - rows:], self.w["final_norm"].double()) @ self.w["lm_head"].double().t()


def exact(case, seed):
    """What run() returns, in 64 bits.  The logits behind a greedy text follow the text that 64-bit arithmetic decodes; sampled
    tokens hang on the library's own random numbers and have no such value."""
    if case["kind"] == "generate" and case["temperature"] > 0.0:
        return None
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    rng = np.random.RandomState(int(seed) % (2**31 - 1))
    w = _weights(case, gen)
    if case["kind"] == "fit":
        tokens = rng.randint(0, case["vocab"], (case["sequences"], case["length"])).astype(np.int32)
        layers = [{n: t.double().requires_grad_(True) for n, t in lw.items()} for lw in w["layers"]]
        trace, fit = np.zeros(case["layers"]), np.zeros(case["layers"])
        for seq in tokens:
            out = _Exact(case, w, grad=True).logits(seq[:-1], len(seq) - 1, layers)
            torch.nn.functional.cross_entropy(out, torch.as_tensor(seq[1:], device="cuda").long()).backward()
            for l, lw in enumerate(layers):
                for t in lw.values():
                    g = float((t.grad * t.grad).sum()) / len(tokens)
                    trace[l] += g
                    fit[l] += g * float((t.detach() * t.detach()).mean())
                    t.grad = None
        return {"trace": trace, "fit": fit}
    with torch.no_grad():
        m = _Exact(case, w)
        if case["kind"] == "score":
            tokens = rng.randint(0, case["vocab"], case["length"]).astype(np.int32)
            out = m.logits(tokens, len(tokens)).cpu().numpy()
            return [out[i:i + 80] for i in range(0, len(tokens), 80)]
        text = list(rng.randint(0, case["vocab"], (case["batch"], case["prompt"])).astype(np.int32)[0])
        last = [m.logits(text, min(TAIL_ROWS, len(text)))]
        for _ in range(case["new"]):
            text.append(int(last[-1][-1].argmax()))
            last.append(m.logits(text[-1:], 1))
        return {"tokens": None, "rounds": None, "logits": torch.cat(last)[-min(TAIL_ROWS, len(text)):].cpu().numpy()}
