"""The work a user of this library has it do, as cases that can be timed and compared.

Three kinds of case, all through the public entry points of `paper_2607_14107_b200.binding`:

  decode     a whole decode of a batch of prompts: `Polestar(...)` (block-entry forward over the prompt, the prefill
             direction), then commit / step until every block is done, tokens back to the host
  refresh    one call chain of the stand-alone cache refresh over the layers of a cache: select the stale rows, gather,
             QKV projection, rotary embedding, scatter
  attention  attention of a set of query rows over a cache, with or without the drift of stored attention rows, over
             the caches of several layers
  confidence argmax and confidence of logits rows

Model widths, prompt / generation / block lengths and refresh fractions are those of `inputs.config` and of the
benchmark, or generic odd sizes around them.

Weights are random, except for a few rows that make the decode decisive, as trained weights do: with plain random
weights every confidence is ~1/vocabulary and the order in which masked positions are committed hangs on the last bit
of two nearly equal numbers.  Here one head of the first layer attends from position i to position i - stride, and the
LM head maps what it copies to a successor token, so a masked position is predicted with high confidence as soon as the
token `stride` places before it is known.  Every forward then commits `stride` tokens by confidence (trained models:
between 1.5 and 3.7 tokens per forward), and all other heads, layers and tokens are random.
"""
import math

import numpy as np
import torch

from paper_2607_14107_b200 import binding as Bd
from paper_2607_14107_b200 import inputs as I

# widths of the models (inputs.config): depth, d_model, heads, kv heads, head_dim, d_ffn, vocab, dtype, eps, rope theta
MODELS = {"llada": "c2", "dream": "c3", "tiny32": "c1", "tiny16": "c1b"}


# ------------------------------------------------------------------------------------------
# cases
# ------------------------------------------------------------------------------------------

def listed():
    return [
        # the benchmark's decode (LLaDA-8B shape, 256 + 256, block 32, one sequence) at about three tokens per forward,
        # refresh steps and plain steps alternating: the interactive, latency-bound use
        dict(name="decode-llada-b1", kind="decode", model="llada", batch=1, prompt=256, gen=256, block=32, stride=3, policy="position"),
        # the same with the paper's default policy: drift on centroid proxies, refresh every step
        dict(name="decode-llada-proxy", kind="decode", model="llada", batch=1, prompt=256, gen=128, block=32, stride=4, policy="proxy"),
        # short, hard-to-parallelise generations (block 8), odd prompt length
        dict(name="decode-llada-short", kind="decode", model="llada", batch=1, prompt=131, gen=32, block=8, stride=2, policy="position"),
        # a batch on the Dream-7B shape (grouped-query attention, wide FFN), 1024 positions
        dict(name="decode-dream-b4", kind="decode", model="dream", batch=4, prompt=896, gen=128, block=32, stride=2, policy="position"),
        # long sequences in a larger batch: 2048 positions, block 64; the largest case
        dict(name="decode-llada-long-b8", kind="decode", model="llada", batch=8, prompt=1984, gen=64, block=64, stride=4, policy="position"),
        # prefill direction: almost all work in block-entry forwards, ragged length (every block is done by its entry)
        dict(name="entry-llada-b3", kind="decode", model="llada", batch=3, prompt=777, gen=64, block=32, stride=32, policy="position"),
        # fp32 model small enough for a laptop's oracle: launches and host work per forward
        dict(name="decode-tiny-fp32", kind="decode", model="tiny32", batch=1, prompt=64, gen=64, block=32, stride=2, policy="position"),
        # refresh micro-benchmark, 1 % of 4096 positions: the smallest refresh, bound by the weight stream
        dict(name="refresh-1pct", kind="refresh", heads="llada", batch=1, positions=4096, frac=0.01, layers=4),
        # ... and a batch of eight at 25 %: 8192 rows, bound by the tensor cores
        dict(name="refresh-b8-25pct", kind="refresh", heads="llada", batch=8, positions=4096, frac=0.25, layers=2),
        # drift + attention of the window and the active block over a 512-position cache, as in every layer of a refresh step
        dict(name="attention-step", kind="attention", heads="llada", rows=128, keys=512, drift=True, layers=8),
        # the same for the block-entry rows of a long sequence (stored rows dominate)
        dict(name="attention-entry", kind="attention", heads="llada", rows=2048, keys=2048, drift=True, layers=2),
        # confidences of one block at the LLaDA vocabulary
        dict(name="confidence-block", kind="confidence", rows=32, vocab=126464),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "refresh", "refresh", "attention", "attention", "confidence"])
    if kind == "decode":
        model = rng.choice(["llada", "llada", "llada", "dream", "dream", "tiny32", "tiny16"])
        batch = rng.choice([1, 1, 1, 2, 3, 4, 6, 8])
        block = rng.choice([8, 16, 24, 32, 32, 48, 64])
        gen = block * rng.randint(1, 3)
        prompt = _log_int(rng, 64, 1900)
        # (the NVFP4 hidden cache only on the fp32 model: next to a code boundary the last bit of a bf16 model's hidden value
        # moves the stored value by a whole code step, and two correct decodes end up 4 % apart)
        policy = rng.choice(["position", "position", "position", "proxy", "nvfp4" if model == "tiny32" else "proxy"])
        # at most 20 forwards: a drawn decode stays below the largest listed one
        stride = max(rng.choice([1, 2, 2, 3, 4, block]), -(-gen // 20))
        return dict(kind="decode", model=model, batch=batch, prompt=prompt, gen=gen, block=block, stride=min(stride, block), policy=policy)
    if kind == "refresh":
        batch = rng.choice([1, 1, 2, 4, 8])
        positions = _log_int(rng, 300, 4096)
        frac = math.exp(rng.uniform(math.log(0.01), 0.0))
        return dict(kind="refresh", heads=rng.choice(["llada", "dream"]), batch=batch, positions=positions, frac=round(frac, 4), layers=2)
    if kind == "attention":
        keys = _log_int(rng, 96, 2048)
        rows = _log_int(rng, 1, keys)
        return dict(kind="attention", heads=rng.choice(["llada", "dream"]), rows=rows, keys=keys, drift=rng.random() < 0.6,
                    layers=8 if rows * keys < 1 << 19 else 2)
    return dict(kind="confidence", rows=_log_int(rng, 1, 512), vocab=2 * _log_int(rng, 500, 76032))


# ------------------------------------------------------------------------------------------
# shapes
# ------------------------------------------------------------------------------------------

def _model(name):
    return I.config(MODELS[name])[0]


def _params(c):
    p = I.Params(batch=c["batch"], prompt_len=c["prompt"], gen_len=c["gen"], block=c["block"], max_steps=c["gen"])
    if c["policy"] != "position":
        p.select_mode = I.SELECT_CLUSTER_TOPK
    if c["policy"] == "nvfp4":
        p.flags |= I.FLAG_NVFP4_HCACHE
    return p


def _forwards(c):
    """(rows that enter a layer, rows that leave it, rows whose attention is recorded, logits rows), per sequence, of every
    forward of a decode that commits `stride` tokens at a time."""
    p = _params(c)
    N, B, out = p.seq_len, p.block, []
    for b in range(p.n_blocks):
        start = p.prompt_len + b * B
        W = min(start, 2 * B) + min(N - start - B, B)
        rec = W if p.select_mode == I.SELECT_TOPK_FRAC else p.n_clusters
        sel = int(p.select_frac * W + 0.5) if p.select_mode == I.SELECT_TOPK_FRAC else W * p.cluster_k // p.n_clusters
        rows = N if b % p.full_entry_period == 0 else B + W
        out.append((rows, rows, rec, B))
        left, cum = B - c["stride"], c["stride"]
        while left > 0:
            if cum > p.tau_upd:
                cum = 0
                out.append((B + W, B + sel, rec, B))
            else:
                out.append((B, B, 0, B))
            left -= c["stride"]
            cum += c["stride"]
    return out


def _heads(c):
    m = _model(c["heads"])
    return m, m.n_heads, m.n_kv_heads, m.head_dim


# ------------------------------------------------------------------------------------------
# state
# ------------------------------------------------------------------------------------------

class _State:
    pass


def _normal(gen, shape, std, dtype):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=gen)


def _decisive_weights(m, stride, gen):
    """Random weights in the library's layout with the copy head described at the top of the file.

    Channels 0 and 1 of the residual stream are reserved: every token carries the same value in channel 0, which only the
    copy head's queries and keys read (so its attention depends on positions alone), and the mask token is nothing but
    channels 0 and 1, so a copied mask predicts nothing.
    """
    dt = I.torch_dtype(m)
    d, half, std = m.d_model, m.head_dim // 2, 0.02
    token_norm = std * math.sqrt(d)
    x0 = math.sqrt(d / 2.0)                                   # channel 0 after RMSNorm
    v_std = std * math.sqrt(d / 2.0)                          # one channel of a copied value
    signal = math.sqrt(m.n_layers)                            # residual channels of the copied signal: as large as all layers' noise
    wo_scale = signal / (std * math.sqrt(m.head_dim) * v_std)
    n_freq = 16
    amp = math.sqrt(80.0 * math.sqrt(m.head_dim) / n_freq) / x0   # peak score of the copy head: 80
    omega = torch.tensor([m.rope_theta ** (-i / half) for i in range(n_freq)], dtype=torch.float64)
    phase = -stride * omega

    def gain():
        g = 1.0 + _normal(gen, (d,), 0.1, torch.float32)
        g[:2] = 1.0
        return g

    packed, copy_v, copy_o = None, None, None
    for l in range(m.n_layers):
        w = {"wq": _normal(gen, (m.d_q, d), std, dt), "wk": _normal(gen, (m.d_kv, d), std, dt), "wv": _normal(gen, (m.d_kv, d), std, dt),
             "wo": _normal(gen, (d, m.d_q), std, dt), "wg": _normal(gen, (m.d_ffn, d), std, dt), "wu": _normal(gen, (m.d_ffn, d), std, dt),
             "wd": _normal(gen, (d, m.d_ffn), std, dt), "norm1": gain(), "norm2": gain()}
        for k in ("wq", "wk", "wv", "wg", "wu"):
            w[k][:, :2] = 0
        w["wo"][:2] = 0
        w["wd"][:2] = 0
        if l == 0:
            w["wq"][:m.head_dim] = 0
            w["wk"][:m.head_dim] = 0
            w["wq"][:n_freq, 0] = (amp * torch.cos(phase)).to("cuda", dt)
            w["wq"][half:half + n_freq, 0] = (amp * torch.sin(phase)).to("cuda", dt)
            w["wk"][:n_freq, 0] = amp
            w["wo"][:, :m.head_dim] *= wo_scale
            copy_v, copy_o = w["wv"][:m.head_dim] * w["norm1"].to(dt), w["wo"][:, :m.head_dim].clone()
        one = dict(layers=[w])
        if l == 0:
            embed = _normal(gen, (m.vocab, d), std, dt)
            embed[:, 0], embed[:, 1] = token_norm, 0.0
            embed[m.mask_id] = 0.0
            embed[m.mask_id, :2] = token_norm
            head = _normal(gen, (m.vocab, d), std, dt)
            # successor of token t: t + 1 (modulo the vocabulary without mask and end token)
            n = m.vocab - 2
            for s in range(0, n, 16384):
                e = min(n, s + 16384)
                sig = ((embed[s:e] @ copy_v.t()) @ copy_o.t()).float()
                sig *= (60.0 if m.n_layers > 8 else 24.0) / math.sqrt(d) / sig.norm(dim=1, keepdim=True)
                to = torch.arange(s + 1, e + 1, device="cuda") % n
                head[to] += sig.to(dt)
            head[:, :2] = 0
            one.update(embed=embed, lm_head=head, final_norm=gain())
        pk = Bd.pack_weights(m, one)
        if packed is None:
            packed = pk
        else:
            for k in ("wqkv", "wo", "w_gate_up", "w_down", "norm1", "norm2"):
                packed[k].extend(pk[k])
    return packed


def prepare(case, seed):
    gen = torch.Generator("cuda").manual_seed(int(seed) * 1000003 + 17)
    s = _State()
    s.case = case
    if case["kind"] == "decode":
        s.m, s.p = _model(case["model"]), _params(case)
        s.packed = _decisive_weights(s.m, case["stride"], gen)
        ids = torch.randint(0, s.m.vocab - 2, (s.p.batch, s.p.prompt_len), generator=gen, device="cuda", dtype=torch.int32)
        s.prompt = ids.cpu().numpy()
        s.logits = torch.empty((s.p.batch, s.p.block, s.m.vocab), dtype=torch.float32, pin_memory=True)
    elif case["kind"] == "refresh":
        m, s.nh, s.nkv, s.dh = _heads(case)
        s.m, b, P, d = m, case["batch"], case["positions"], m.d_model
        s.k = max(1, I.refresh_count(case["frac"], P))
        s.layers = []
        for _ in range(case["layers"]):
            # hidden rows ~ N(0, 1), drift lognormal, as in the refresh micro-benchmark
            s.layers.append(dict(h=_normal(gen, (b, P, d), 1.0, torch.bfloat16), drift=_normal(gen, (b, P), 1.0, torch.float32).exp_(),
                                 w=Bd.tile_major(_normal(gen, (m.d_q + 2 * m.d_kv, d), 0.02, torch.bfloat16)),
                                 norm=1.0 + _normal(gen, (d,), 0.1, torch.float32),
                                 kc=torch.zeros((b, P, m.d_kv), dtype=torch.bfloat16, device="cuda"),
                                 vc=torch.zeros((b, P, m.d_kv), dtype=torch.bfloat16, device="cuda")))
        s.full = torch.zeros((b, P), dtype=torch.int32, device="cuda")
        s.idx = torch.zeros((b, s.k), dtype=torch.int32, device="cuda")
        s.count = torch.zeros(b, dtype=torch.int32, device="cuda")
        raw = torch.empty(Bd.polestar_k_refresh_scratch_bytes(b, s.k, d, s.nh, s.nkv, s.dh) + 1024, dtype=torch.uint8, device="cuda")
        s.scratch = raw[(-raw.data_ptr()) % 1024:]
    elif case["kind"] == "attention":
        m, s.nh, s.nkv, s.dh = _heads(case)
        R, N = case["rows"], case["keys"]
        s.layers = []
        for _ in range(case["layers"]):
            # score spread sigma ~ 1.6 over the keys, what the random-weight models show; the stored row is another query's
            q, k = _normal(gen, (R, m.d_q), 1.27, torch.bfloat16), _normal(gen, (N, m.d_kv), 1.27, torch.bfloat16)
            v = _normal(gen, (N, m.d_kv), 1.0, torch.bfloat16)
            a = dict(q=q, k=k, v=v, prev=None, lse=None, kl=None, out=torch.empty((R, m.d_q), dtype=torch.bfloat16, device="cuda"))
            if case["drift"]:
                a["prev"] = _normal(gen, (R, s.nh, N), 1.6, torch.float32)
                a["lse"] = torch.logsumexp(a["prev"], -1)
                a["kl"] = torch.empty((R, s.nh), dtype=torch.float32, device="cuda")
            s.layers.append(a)
    else:
        R, V = case["rows"], case["vocab"]
        s.logits = _normal(gen, (R, V), 1.5, torch.float32)
        s.logits[torch.arange(R, device="cuda"), torch.randint(0, V - 2, (R,), generator=gen, device="cuda")] += 12.0   # a decided row
        s.mask = V - 1
        s.yhat = torch.zeros(R, dtype=torch.int32, device="cuda")
        s.conf = torch.zeros(R, dtype=torch.float32, device="cuda")
        s.scratch = torch.empty(R * 512, dtype=torch.uint8, device="cuda")
    return s


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------

def run(s):
    kind = s.case["kind"]
    if kind == "decode":
        dec = Bd.Polestar(s.m, s.packed, s.p, s.prompt)
        dec.decode()
        tokens = dec.tokens()
        # logits of the last forward into a page-locked buffer (`Polestar.read` would allocate a pageable one)
        Bd._check(Bd.load().polestar_read(dec.ctx, Bd.READ_LOGITS, 0, s.logits.data_ptr(), s.logits.numel() * 4))
        dec.destroy()
        return {"tokens": tokens, "logits": s.logits}
    if kind == "refresh":
        for l in s.layers:
            Bd.polestar_k_select(l["drift"], I.SELECT_TOPK_COUNT, s.k, 0.0, 0.0, s.full, s.count)
            s.idx.copy_(s.full[:, :s.k])
            Bd.polestar_k_refresh(l["h"], s.idx, s.count, l["w"], l["norm"], l["kc"], l["vc"], None, s.k, s.nh, s.nkv, s.dh,
                                  s.m.rms_eps, s.m.rope_theta, s.scratch)
        return {"idx": s.idx, "count": s.count, "k": [l["kc"] for l in s.layers], "v": [l["vc"] for l in s.layers]}
    if kind == "attention":
        for l in s.layers:
            Bd.polestar_k_attention(l["q"], l["k"], l["v"], l["prev"], l["lse"], l["kl"], l["out"], s.nh, s.nkv, s.dh)
        return {n: [l[n] for l in s.layers] for n in ("out", "prev", "lse", "kl") if s.layers[0][n] is not None}
    Bd.polestar_k_confidence(s.logits, s.mask, s.yhat, s.conf, s.scratch)
    return {"yhat": s.yhat, "conf": s.conf}


# ------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far two correct implementations are apart
# ------------------------------------------------------------------------------------------

def work(case):
    if case["kind"] == "decode":
        m, p = _model(case["model"]), _params(case)
        es = 2 if m.dtype == I.DTYPE_BF16 else 4
        d, dq, dkv, F, V, L, bs, N = m.d_model, m.d_q, m.d_kv, m.d_ffn, m.vocab, m.n_layers, p.batch, p.seq_len
        n_in, n_out = (dq + 2 * dkv) * d, d * dq + 3 * d * F
        by = fl = 0
        for rows_in, rows_out, rec, head in _forwards(case):
            by += (L * (n_in + n_out) + V * d) * es + 2 * L * bs * N * dkv * es + 2 * L * bs * rec * m.n_heads * N * 4 + bs * head * V * 4
            fl += 2 * bs * (L * (rows_in * n_in + rows_out * n_out) + head * V * d) + 4 * L * bs * rows_in * N * dq
        return {"bytes": by, "flops": fl}
    if case["kind"] == "refresh":
        m, nh, nkv, dh = _heads(case)
        rows = case["batch"] * max(1, I.refresh_count(case["frac"], case["positions"]))
        n = m.d_q + 2 * m.d_kv
        by = n * m.d_model * 2 + rows * (m.d_model + 2 * m.d_kv) * 2 + case["batch"] * case["positions"] * 4
        return {"bytes": case["layers"] * by, "flops": case["layers"] * 2 * rows * n * m.d_model}
    if case["kind"] == "attention":
        m, nh, nkv, dh = _heads(case)
        R, N = case["rows"], case["keys"]
        by = 2 * N * m.d_kv * 2 + 2 * R * m.d_q * 2 + (R * nh * (2 * N + 3) * 4 if case["drift"] else 0)
        return {"bytes": case["layers"] * by, "flops": case["layers"] * 4 * R * N * m.d_q}
    return {"bytes": case["rows"] * (case["vocab"] * 4 + 8), "flops": 3 * case["rows"] * case["vocab"]}


def tolerance(case):
    if case["kind"] == "confidence":
        return {"rel": 1e-5}
    if case["kind"] == "decode":
        # bf16: two runs of one build, whose projections are added up in another order, end 0.4 - 0.7 % apart in the logits
        if case["model"] == "tiny32":
            return {"rel": 1e-2 if case["policy"] == "nvfp4" else 2e-5}
        return {"rel": 2e-2, "max": 0.2}
    # one bf16 rounding of the operands and one of the result: 0.2 % from a 64-bit computation
    return {"rel": 5e-3, "max": 0.1}
