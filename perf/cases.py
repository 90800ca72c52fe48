"""The work that users of this library have it do, as measurable cases through its public entry
points: single projections (jf_op_gemm), single decoder layers over a paged cache, prompt prefill,
one Jacobi step with multi-block drafts and a recycled candidate, and whole generations.

Sizes are those of the model shapes in paper_2512_14681_gb300/inputs.py and of bench.py's workloads,
or generic odd ones between them. Single layers are one-layer models of those shapes with a
4,096-token vocabulary and N(0, 0.02) weights. Whole models use tied embeddings and N(0, 5e-4)
weights: their residual stream stays close to the embedding, so the next token (a copy of the last
one) is as decided as a trained model's, where N(0, 0.02) weights leave it to rounding.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2512_14681_gb300 import _lib as J
from paper_2512_14681_gb300 import inputs as I
from paper_2512_14681_gb300.jacobi import Context, Gen, op_gemm

LAYER_STD = 0.02
MODEL_STD = 5e-4
LAYER_VOCAB = 4096

SHAPES = {
    "7b-layer": dataclasses.replace(I.QWEN7B_BF16, name="7b-layer", n_layers=1, vocab=LAYER_VOCAB),
    "1.5b-layer": dataclasses.replace(I.QWEN15B_BF16, name="1.5b-layer", n_layers=1, vocab=LAYER_VOCAB),
    "7b": dataclasses.replace(I.QWEN7B_BF16, name="7b-tied", tie_embeddings=True),
    "1.5b": I.QWEN15B_BF16,
    "tiny": I.TINY_F32,
}


def listed():
    return [
        # one projection of a decode forward (the 7B QKV matrix, a 32-token block): the smallest call,
        # where launch and latency count as much as the weight stream
        dict(name="proj-qkv-32", kind="proj", N=4608, K=3584, M=32, bf16=True),
        # a projection of no tile's size: odd feature count, K not a multiple of 64, odd rows
        dict(name="proj-ragged-77", kind="proj", N=3001, K=1544, M=77, bf16=True),
        # the 7B gate/up matrix over a 512-row prefill chunk: tensor-bound
        dict(name="proj-gateup-512", kind="proj", N=37888, K=3584, M=512, bf16=True),
        # a projection of the small fp32 models (CUDA cores)
        dict(name="proj-f32-40", kind="proj", N=4096, K=1024, M=40, bf16=False),
        # one 7B decoder layer, a 32-token draft over a 1,024-token cache: the headline decode iteration
        dict(name="layer-7b-p1024-n32", kind="layer", shape="7b-layer", P=1024, n=32),
        # one 7B decoder layer, a 128-token draft over a long cache: attention-bound
        dict(name="layer-7b-p32768-n128", kind="layer", shape="7b-layer", P=32768, n=128),
        # one 1.5B decoder layer with odd sizes: every launch is latency-bound
        dict(name="layer-1.5b-p777-n19", kind="layer", shape="1.5b-layer", P=777, n=19),
        # prompt prefill through one 7B layer in 512-row forwards, the last one partial
        dict(name="prefill-7b-4000", kind="prefill", shape="7b-layer", P=4000, n=8, rows=512),
        # one Jacobi step of the whole 7B model: four 32-token blocks and one recycled candidate
        dict(name="step-7b-4x32-cand", kind="step", shape="7b", P=2048, block=32, blocks=4, cands=1),
        # whole generation, 7B: prefill and block-sequential Jacobi decoding at batch 1
        dict(name="generate-7b", kind="generate", shape="7b", prompts="1024", blocks="32", join="0", p=0.3, new=128),
        # serving on the 1.5B model: four sequences with their own block sizes, one joining late
        dict(name="serve-1.5b-4seq", kind="generate", shape="1.5b", prompts="512 301 1200 640",
             blocks="16 8 32 11", join="0 0 0 3", p=0.5, new=64),
        # whole generation of the tiny fp32 model (prompt 32, block 8, 64 tokens): launch-bound
        dict(name="generate-tiny-f32", kind="generate", shape="tiny", prompts="32", blocks="8", join="0", p=-1.0,
             new=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _text(values):
    return " ".join(str(v) for v in values)


def _ints(text):
    """Per-sequence numbers of a case ("512 301")."""
    return [int(v) for v in text.split()]


def draw(rng):
    kind = rng.choice(["proj", "proj", "layer", "layer", "layer", "prefill", "step", "generate"])
    if kind == "proj":
        bf16 = rng.random() < 0.8
        return dict(kind="proj", N=_log_int(rng, 512, 37888 if bf16 else 4096),
                    K=8 * _log_int(rng, 32, 2368 if bf16 else 128), M=_log_int(rng, 1, 512 if bf16 else 64), bf16=bf16)
    if kind == "layer":
        return dict(kind="layer", shape=rng.choice(["7b-layer", "1.5b-layer"]), P=_log_int(rng, 64, 32768),
                    n=_log_int(rng, 1, 256))
    if kind == "prefill":
        return dict(kind="prefill", shape=rng.choice(["7b-layer", "1.5b-layer"]), P=_log_int(rng, 64, 8192),
                    n=rng.randint(1, 16), rows=rng.choice([128, 256, 512, 1000]))
    if kind == "step":
        return dict(kind="step", shape="1.5b", P=_log_int(rng, 64, 8192), block=_log_int(rng, 4, 64),
                    blocks=rng.randint(1, 4), cands=rng.randint(0, 4))
    n = rng.randint(1, 4)
    return dict(kind="generate", shape="1.5b", prompts=_text(_log_int(rng, 64, 2048) for _ in range(n)),
                blocks=_text(_log_int(rng, 2, 64) for _ in range(n)),
                join=_text(rng.choice([0, 0, 2, 5]) if b else 0 for b in range(n)), p=rng.choice([0.1, 0.3, 0.5, 0.7]),
                new=rng.randint(16, 64))


def _tokens(vocab, n, *key):
    return np.random.default_rng(key).integers(0, vocab, size=n, dtype=np.int64).astype(np.int32)


def _proj_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.bfloat16 if case["bf16"] else torch.float32
    W = (torch.randn(case["N"], case["K"], generator=g, device="cuda") * LAYER_STD).to(dt)
    X = torch.randn(case["M"], case["K"], generator=g, device="cuda").to(dt)
    return W, X


def _std(case):
    return MODEL_STD if case["kind"] in ("step", "generate") and case["shape"] != "tiny" else LAYER_STD


def _draft_len(case):
    return case["block"] * case["blocks"], case["block"] * case["cands"]


def prepare(case, seed):
    if case["kind"] == "proj":
        W, X = _proj_inputs(case, seed)
        return dict(kind="proj", W=W, X=X)
    shape = SHAPES[case["shape"]]
    kind = case["kind"]
    if kind in ("layer", "prefill"):
        P, n = case["P"], case["n"]
        rows = case.get("rows", 512)
        ctx = Context(shape, max_ctx=P + n + 32, max_rows=max(rows, n))
        ctx.init_random_weights(seed, LAYER_STD)
        toks = _tokens(shape.vocab, P + n, seed, 1)
        if kind == "layer":
            ctx.prefill(0, toks[:P])
        return dict(kind=kind, ctx=ctx, prompt=toks[:P], draft=toks[P:])
    if kind == "step":
        P = case["P"]
        main, cand = _draft_len(case)
        ctx = Context(shape, max_ctx=P + main + 32, max_rows=max(512, main + cand))
        ctx.init_random_weights(seed, _std(case))
        toks = _tokens(shape.vocab, P + main + cand, seed, 1)
        ctx.prefill(0, toks[:P])
        n, K = case["block"], case["blocks"]
        blocks = [(J.JF_BLOCK_RA, P, n, -1)]
        blocks += [(J.JF_BLOCK_PSEUDO, P + b * n, n, b - 1) for b in range(1, K)]
        blocks += [(J.JF_BLOCK_CAND, P, n, -1)] * case["cands"]
        return dict(kind=kind, ctx=ctx, P=P, blocks=blocks, draft=toks[P:])
    lens, sizes = _ints(case["prompts"]), _ints(case["blocks"])
    S = len(lens)
    new, n = case["new"], max(sizes)
    ctx = Context(shape, max_seqs=S, max_ctx=max(lens) + new + 2 * n + 64, max_rows=max(512, 64 * S + sum(sizes)),
                  logits_rows=1)
    ctx.init_random_weights(seed, _std(case))
    prompts = [_tokens(shape.vocab, L, seed, 1, b) for b, L in enumerate(lens)]
    inject = case["p"] >= 0
    gen = Gen(block_size=n, init="inject" if inject else "repeat", inject_p=max(case["p"], 0.0), seed=I.INJECT_SEED,
              max_new=new, block_sizes=tuple(sizes), join_iters=tuple(_ints(case["join"])))
    # the greedy continuation that injected drafts are taken from: these models copy the last token
    truth = np.stack([np.full(new + 2 * n + 2, p[-1], dtype=np.int32) for p in prompts]) if inject else None
    return dict(kind=kind, ctx=ctx, prompts=prompts, gen=gen, truth=truth)


def run(state):
    kind = state["kind"]
    if kind == "proj":
        return op_gemm(state["W"], state["X"])[0]
    ctx = state["ctx"]
    if kind == "layer":
        return ctx.forward_logits(0, state["draft"], want_logits=False)[1]
    if kind == "prefill":  # a new prompt into the sequence's slot, then the rows that follow it
        ctx.truncate(0, 0)
        ctx.prefill(0, state["prompt"])
        return ctx.forward_logits(0, state["draft"], want_logits=False)[1]
    if kind == "step":  # verify a draft, then roll back as a caller that tries another one does
        out = ctx.jacobi_step(0, state["blocks"], state["draft"])
        ctx.truncate(0, state["P"])
        return [out["counts"], out["committed"], out["predictions"], out["top2"]]
    # decode, then score the next position from the cache that decoding left
    out = ctx.generate(state["prompts"], state["gen"], truth=state["truth"])
    logits = ctx.forward_logits(0, out.tokens[0, -1:], want_hidden=False)[0]
    return [out.tokens, out.iterations, logits]


def _iterations(n, p, new):
    """Expected iterations for `new` tokens in blocks of n whose draft tokens are wrong at rate p."""
    if p < 0:
        return new
    f = [0.0] * (n + 1)
    for L in range(1, n + 1):
        f[L] = 1.0 + sum((1 - p) ** (k - 1) * (p if k < L else 1.0) * f[L - k] for k in range(1, L + 1))
    return f[n] * new / n


def _forward_work(shape, rows, keys):
    """(weight and cache bytes, flops) of one forward of `rows` rows seeing `keys` keys each."""
    w = shape.weight_bytes()
    es = 2 if shape.bf16 else 4
    mm = 2.0 * rows * w / es
    at = 4.0 * rows * keys * shape.n_heads * shape.head_dim * shape.n_layers
    return w + keys * shape.kv_bytes_per_token(), mm + at


def work(case):
    if case["kind"] == "proj":
        N, K, M = case["N"], case["K"], case["M"]
        es = 2 if case["bf16"] else 4
        return dict(bytes=es * (N * K + M * K) + 4 * M * N, flops=2.0 * M * N * K)
    shape = SHAPES[case["shape"]]
    if case["kind"] == "layer":
        b, f = _forward_work(shape, case["n"], case["P"] + case["n"] // 2)
        return dict(bytes=b + 4 * case["n"] * shape.d_model, flops=f)
    if case["kind"] == "prefill":
        b, f = _forward_work(shape, case["P"], case["P"] // 2)
        b2, f2 = _forward_work(shape, case["n"], case["P"])
        return dict(bytes=b + b2 + 4 * case["n"] * shape.d_model, flops=f + f2)
    if case["kind"] == "step":
        main, cand = _draft_len(case)
        b, f = _forward_work(shape, main + cand, case["P"])
        return dict(bytes=b, flops=f)
    # all sequences share each iteration's weight stream; their expected lengths differ little
    its = [_iterations(n, case["p"], case["new"]) for n in _ints(case["blocks"])]
    bytes_ = flops = 0.0
    for L, n, it in zip(_ints(case["prompts"]), _ints(case["blocks"]), its):
        b, f = _forward_work(shape, L, L // 2)
        bytes_ += b
        flops += f + it * _forward_work(shape, n / 2, L)[1]
        bytes_ += it * L * shape.kv_bytes_per_token()
    return dict(bytes=bytes_ + max(its) * shape.weight_bytes(), flops=flops)


def tolerance(case):
    if case["kind"] == "proj":
        # fp32 sums of K products: 3.8e-6 from the 64-bit result at K = 3584 unsplit, growing with K
        return {"rel": 1.5e-5 * max(1.0, case["K"] / 3584)}
    if case["kind"] in ("layer", "prefill"):
        # bf16 activations between the layer's matrices: 3e-3 between two orders of the split-K sums
        return {"rel": 1.2e-2}
    if case["shape"] == "tiny":
        return {"rel": 1e-5, "differ": 0.0}
    # 28 layers of bf16 activations: 3.5e-3 between two orders of the split-K sums; the tokens are
    # decided by wide margins
    return {"rel": 1.4e-2, "differ": 0.0}


# ---------------------------------------------------------------------------------------------
# 64-bit results in plain torch. The weights are drawn from their published definition: SplitMix64
# keyed by (seed, tensor id), Box-Muller on outputs 2j and 2j+1, rounded to the model's type.
# ---------------------------------------------------------------------------------------------
def _signed(v):
    return v - (1 << 64) if v >= 1 << 63 else v


def _shr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _splitmix(s, i):
    z = s + (i + 1) * _signed(0x9E3779B97F4A7C15)
    z = (z ^ _shr(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _signed(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _tensor(shape, seed, std, tid, rows, cols):
    one = torch.tensor
    s = _splitmix(one(seed, device="cuda"), one(tid, device="cuda"))
    n = rows * cols
    j = torch.arange((n + 1) // 2, device="cuda")
    u1 = (_shr(_splitmix(s, 2 * j), 11).double() + 1.0) / 2.0 ** 53
    u2 = _shr(_splitmix(s, 2 * j + 1), 11).double() / 2.0 ** 53
    r, a = std * torch.sqrt(-2.0 * torch.log(u1)), 2.0 * math.pi * u2
    w = torch.stack([r * torch.cos(a), r * torch.sin(a)], 1).reshape(-1)[:n].reshape(rows, cols)
    return w.to(torch.bfloat16 if shape.bf16 else torch.float32).double()


def _rms(x, eps):
    return x / torch.sqrt(torch.mean(x * x, -1, keepdim=True) + eps)


def _rope(x, pos, theta):
    half = x.shape[-1] // 2
    ang = pos[:, None].double() * theta ** (-torch.arange(half, device="cuda").double() / half)
    c, s = torch.cos(ang)[:, None], torch.sin(ang)[:, None]
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * c - b * s, b * c + a * s], -1)


class _Model64:
    """The decoder in 64 bits, no rounding between its matrices."""

    def __init__(self, shape, seed, std):
        d, hd, Hq, Hkv, F = shape.d_model, shape.head_dim, shape.n_heads, shape.n_kv_heads, shape.d_ff
        self.s = shape
        t = lambda tid, r, c: _tensor(shape, seed, std, tid, r, c)
        self.E = t(0, shape.vocab, d)
        self.layers = []
        for l in range(shape.n_layers):
            o = 8 + 16 * l
            w = dict(q=t(o + 1, Hq * hd, d), k=t(o + 2, Hkv * hd, d), v=t(o + 3, Hkv * hd, d), o=t(o + 4, d, Hq * hd),
                     g=t(o + 6, F, d), u=t(o + 7, F, d), dn=t(o + 8, d, F))
            if shape.qkv_bias:
                w.update(bq=t(o + 9, 1, Hq * hd), bk=t(o + 10, 1, Hkv * hd), bv=t(o + 11, 1, Hkv * hd))
            self.layers.append(w)

    def hidden(self, tokens, last):
        """Residual stream of the last `last` rows after every layer (causal)."""
        s = self.s
        n = len(tokens)
        G = s.n_heads // s.n_kv_heads
        x = self.E[torch.as_tensor(tokens, device="cuda").long()]
        pos = torch.arange(n, device="cuda")
        for i, w in enumerate(self.layers):
            keep = last if i == len(self.layers) - 1 else n
            h = _rms(x, s.rms_eps)
            x, hq, pq = x[n - keep:], h[n - keep:], pos[n - keep:]
            q, k, v = hq @ w["q"].T, h @ w["k"].T, h @ w["v"].T
            if s.qkv_bias:
                q, k, v = q + w["bq"], k + w["bk"], v + w["bv"]
            q = _rope(q.view(keep, s.n_heads, s.head_dim), pq, s.rope_theta)
            k = _rope(k.view(n, s.n_kv_heads, s.head_dim), pos, s.rope_theta)
            v = v.view(n, s.n_kv_heads, s.head_dim)
            masked = pos[None, :] > pq[:, None]
            heads = []
            for hh in range(s.n_heads):
                sc = (q[:, hh] @ k[:, hh // G].T / math.sqrt(s.head_dim)).masked_fill(masked, -math.inf)
                heads.append(torch.softmax(sc, -1) @ v[:, hh // G])
            x = x + torch.cat(heads, 1) @ w["o"].T
            h = _rms(x, s.rms_eps)
            g, u = h @ w["g"].T, h @ w["u"].T
            x = x + (g / (1.0 + torch.exp(-g)) * u) @ w["dn"].T
        return x


def exact(case, seed):
    if case["kind"] == "proj":
        W, X = _proj_inputs(case, seed)
        return X.double() @ W.double().T
    if case["kind"] == "step" or case["shape"] in ("7b", "1.5b"):
        return None  # 28 layers in 64 bits
    shape = SHAPES[case["shape"]]
    m = _Model64(shape, seed, LAYER_STD)
    if case["kind"] in ("layer", "prefill"):
        toks = _tokens(shape.vocab, case["P"] + case["n"], seed, 1)
        return m.hidden(toks, case["n"]).cpu().numpy()
    head = _tensor(shape, seed, LAYER_STD, 1, shape.vocab, shape.d_model)
    toks = _tokens(shape.vocab, _ints(case["prompts"])[0], seed, 1, 0).tolist()
    for _ in range(case["new"]):
        toks.append(int(torch.argmax(_rms(m.hidden(toks, 1), shape.rms_eps) @ head.T)))
    return [np.array([toks[-case["new"]:]], dtype=np.int32), None, None]
