"""Performance cases of the public entry points: the work that a program using this library has it do.

Three families, each over its real range of sizes:

* the sublayer building blocks, ``fused_gemv`` (one to nine activation rows: a decode step, a draft step, the rows
  of a verification) and ``gemm_bf16`` (the dense product of a prompt);
* the prompt pass, ``Decoder.prefill``, of decoders with the widths of the benchmark shapes and a few layers;
* decoding on top of a filled KV cache: draft steps under a skip mask, verify passes, and one whole session of the
  tiny decoder, with the tokens supplied by the caller (as when drafts come from elsewhere), so that a change of
  rounding never sends two runs down different texts.

Vocabularies are in proportion to the number of layers (32000 for 32 layers), so that the LM head keeps the share of
a pass that it has in the full decoder.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2410_01028_b200 as asd
from synth import LLAMA_13B, LLAMA_7B, TINY, DecoderShape

_EPS, _THETA, _STD = 1e-5, 10000.0, 0.02
_EPI = {"plain": asd.EPI_PLAIN, "swiglu": asd.EPI_SWIGLU, "residual": asd.EPI_RESIDUAL}


# ---------------------------------------------------------------- the cases
def _gemv(rows, n_in, n_rows, epi, norm):
    return {"kind": "gemv", "rows": rows, "n_in": n_in, "n_rows": n_rows, "epi": epi, "norm": norm}


def _gemm(m, n, k):
    return {"kind": "gemm", "m": m, "n": n, "k": k}


def _decoder(kind, shape, layers, prompt, **more):
    vocab = shape.vocab * layers // shape.n_layers
    return {"kind": kind, "layers": layers, "d_model": shape.d_model, "heads": shape.n_heads, "kv_heads": shape.kv_heads,
            "head_dim": shape.head_dim, "d_ffn": shape.d_ffn, "vocab": vocab, "prompt": prompt, **more}


# grouped queries and the smaller head size of the dense prompt path
_GQA64 = DecoderShape(n_layers=32, d_model=2048, n_heads=32, head_dim=64, d_ffn=5504, vocab=32000, n_kv_heads=8)


def listed():
    return [
        # the smallest call: one decode row through the QKV projection of a narrow decoder; latency counts
        dict(_gemv(1, 2048, 6144, "plain", True), name="gemv_qkv_2048_1row"),
        # one decode row through the gate/up projection of the 7B width: the largest weight stream of a layer
        dict(_gemv(1, 4096, 22016, "swiglu", True), name="gemv_gateup_4096_1row"),
        # the five rows of a verification with four drafts through a down projection with residual add and cosine
        dict(_gemv(5, 13760, 5120, "residual", False), name="gemv_down_5120_5rows"),
        # nine rows (eight drafts) through a matrix of odd sizes
        dict(_gemv(9, 2056, 6145, "plain", True), name="gemv_ragged_9rows"),
        # the QKV product of an ordinary prompt, and the gate/up product of a full chunk of a long one
        dict(_gemm(511, 12288, 4096), name="gemm_qkv_511"),
        dict(_gemm(2048, 22016, 4096), name="gemm_gateup_2048"),
        # an ordinary prompt, a long one (four chunks; attention is most of it), and an odd one with grouped queries
        dict(_decoder("prefill", LLAMA_7B, 4, 512), name="prefill_7b_512"),
        dict(_decoder("prefill", LLAMA_7B, 2, 8192), name="prefill_7b_8192"),
        dict(_decoder("prefill", _GQA64, 4, 1023), name="prefill_gqa64_1023"),
        # a round of draft steps under a skip mask
        dict(_decoder("draft", LLAMA_7B, 4, 512, steps=8, skip=True), name="draft_7b_512"),
        # a long prompt followed by rounds of verification on top of it
        dict(_decoder("verify", LLAMA_7B, 2, 8192, rounds=16, rows=5), name="verify_7b_8192"),
        # the tiny decoder, whole: prompt, then rounds of four draft steps and one verify pass; every pass is latency
        dict(_decoder("session", TINY, 4, 32, rounds=6, rows=5, skip=True), name="tiny_session"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gemv", "gemv", "gemm", "gemm", "prefill", "prefill", "draft", "verify", "session"])
    if kind == "gemv":
        rows, n_in = rng.randint(1, 9), 8 * _log_int(rng, 128, 2752)
        n_rows = _log_int(rng, 1024, min(44032, (180 << 20) // n_in))
        epi = rng.choice(["plain", "swiglu", "residual"])
        return _gemv(rows, n_in, 2 * (n_rows // 2) if epi == "swiglu" else n_rows, epi, epi != "residual" and n_in * rows <= 49152)
    if kind == "gemm":
        m, k = _log_int(rng, 33, 2048), 8 * _log_int(rng, 128, 1376)
        return _gemm(m, _log_int(rng, 1024, 22016), k)
    if kind == "session":
        return _decoder("session", TINY, 4, rng.randint(2, 96), rounds=rng.randint(2, 6), rows=rng.randint(1, 9), skip=rng.random() < 0.5)
    shape = rng.choice([LLAMA_7B, LLAMA_13B, _GQA64])
    if kind == "prefill":
        return _decoder("prefill", shape, rng.randint(1, 2), _log_int(rng, 2, 4096))
    if kind == "draft":
        return _decoder("draft", shape, 2, _log_int(rng, 33, 8192), steps=rng.randint(1, 8), skip=rng.random() < 0.5)
    return _decoder("verify", shape, 2, _log_int(rng, 33, 4096), rounds=rng.randint(4, 16), rows=rng.randint(1, 9))


# ---------------------------------------------------------------- inputs
def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(1000003 * (seed % (1 << 40)) + stream)


def _normal(shape, seed, stream, std=1.0, mean=0.0, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=torch.float32, device="cuda").normal_(mean, std, generator=_gen(seed, stream)).to(dtype)


def _shape(case):
    return DecoderShape(case["layers"], case["d_model"], case["heads"], case["head_dim"], case["d_ffn"], case["vocab"], case["kv_heads"])


class _Weights:
    """Random-init decoder: N(0, 0.02^2), output projections of every sublayer scaled by a factor from U[0.05, 1]."""

    def __init__(self, case, seed):
        s = _shape(case)
        L, d, f, V, kv = s.n_layers, s.d_model, s.d_ffn, s.vocab, s.kv_dim
        scales = 0.05 + 0.95 * torch.rand(2 * L, device="cuda", generator=_gen(seed, 1))
        self.embed, self.lm_head = _normal((V, d), seed, 2, _STD), _normal((V, d), seed, 3, _STD)
        self.final_norm = _normal((d,), seed, 4, _STD, 1.0)
        self.attn_norm, self.mlp_norm = _normal((L, d), seed, 5, _STD, 1.0), _normal((L, d), seed, 6, _STD, 1.0)
        self.wq, self.wk, self.wv = _normal((L, d, d), seed, 7, _STD), _normal((L, kv, d), seed, 8, _STD), _normal((L, kv, d), seed, 9, _STD)
        self.wg, self.wu = _normal((L, f, d), seed, 10, _STD), _normal((L, f, d), seed, 11, _STD)
        self.wo = (_normal((L, d, d), seed, 12, _STD, dtype=torch.float32) * scales[0::2, None, None]).to(torch.bfloat16)
        self.wd = (_normal((L, d, f), seed, 13, _STD, dtype=torch.float32) * scales[1::2, None, None]).to(torch.bfloat16)

    def on_host(self):
        class Host:
            pass

        h = Host()
        for name, t in vars(self).items():
            setattr(h, name, t.view(torch.int16).cpu().numpy().view(np.uint16))
        return h


def _tokens(case, seed):
    """The prompt, and the tokens of the steps after it: [steps] or [rounds, rows] (row 0 committed, the rest drafts)."""
    rng = np.random.default_rng([seed, 77])
    prompt = rng.integers(0, case["vocab"], case["prompt"], dtype=np.int32)
    if case["kind"] == "draft":
        return prompt, rng.integers(0, case["vocab"], case["steps"], dtype=np.int32)
    if case["kind"] in ("verify", "session"):
        return prompt, rng.integers(0, case["vocab"], (case["rounds"], case["rows"]), dtype=np.int32)
    return prompt, None


def _mask(case):
    """Every other attention sublayer and the last MLP sublayer removed, or nothing."""
    a, m = np.zeros(case["layers"], np.uint8), np.zeros(case["layers"], np.uint8)
    if case.get("skip"):
        a[1::2], m[-1] = 1, 1
    return a, m


def prepare(case, seed):
    st = dict(case=case)
    if case["kind"] == "gemv":
        rows, n_in, n_rows, epi = case["rows"], case["n_in"], case["n_rows"], case["epi"]
        st["W"] = _normal((n_rows, n_in), seed, 1, _STD)
        st["x"] = _normal((rows, n_in), seed, 2, dtype=torch.float32 if case["norm"] else torch.bfloat16)
        st["gain"] = _normal((n_in,), seed, 3, _STD, 1.0) if case["norm"] else None
        st["hidden"] = _normal((rows, n_rows), seed, 4, dtype=torch.float32) if epi == "residual" else None
        st["out"] = torch.empty((rows, n_rows // 2), dtype=torch.bfloat16, device="cuda") if epi == "swiglu" else \
            torch.empty((rows, n_rows), dtype=torch.float32, device="cuda")
        st["cos"] = torch.empty(rows, dtype=torch.float32, device="cuda") if epi == "residual" else None
        st["scratch"] = torch.zeros(asd.fused_gemv_scratch_bytes(), dtype=torch.uint8, device="cuda")
        return st
    if case["kind"] == "gemm":
        st["A"], st["W"] = _normal((case["m"], case["k"]), seed, 1), _normal((case["n"], case["k"]), seed, 2, _STD)
        st["C"] = torch.empty((case["m"], case["n"]), dtype=torch.float32, device="cuda")
        st["status"] = torch.zeros(8, dtype=torch.int32, device="cuda")
        return st
    st["prompt"], st["tokens"] = _tokens(case, seed)
    st["mask"] = _mask(case)
    room = 0 if st["tokens"] is None else st["tokens"].size
    dec = st["dec"] = asd.Decoder(_shape(case), max_seq=case["prompt"] + room + 16, max_draft=8, rms_eps=_EPS, rope_theta=_THETA)
    dec.load_weights_host(_Weights(case, seed).on_host())
    dec.set_debug(record_logits=True)
    if case["kind"] == "draft":
        dec.prefill(st["prompt"])
    return st


# ---------------------------------------------------------------- one pass
def _kv_of_last(dec, case):
    rows = [dec.get_kv(layer, case["prompt"] - 1) for layer in range(case["layers"])]
    return [(np.stack(r).astype(np.uint32) << 16).view(np.float32) for r in rows]


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "gemv":
        if st["hidden"] is not None:
            st["out"].copy_(st["hidden"])  # the hidden state that the sublayer's output is added to
        asd.fused_gemv(st["x"], st["W"], _EPI[case["epi"]], st["out"], gain=st["gain"], eps=_EPS, cos=st["cos"], scratch=st["scratch"])
        return [st["out"]] if st["cos"] is None else [st["out"], st["cos"]]
    if kind == "gemm":
        asd.gemm_bf16(st["A"], st["W"], st["C"], st["status"])
        return st["C"]
    dec, logits = st["dec"], []
    if kind == "draft":
        dec.set_skip_mask(*st["mask"])  # installs the draft model; back to the committed length
        for t in st["tokens"]:
            dec.draft_step(int(t))
            logits.append(dec.get_last_logits())
        return {"logits": logits}
    dec.reset()
    dec.prefill(st["prompt"])
    c_attn, c_mlp, _ = dec.get_similarity()
    if kind == "prefill":
        return {"logits": dec.get_last_logits()[-1], "c_attn": c_attn, "c_mlp": c_mlp, "kv": _kv_of_last(dec, case)}
    if kind == "session":
        dec.set_skip_mask(*st["mask"])
    for tokens in st["tokens"]:
        if kind == "session":
            for t in tokens[:-1]:
                dec.draft_step(int(t))
                logits.append(dec.get_last_logits())
        dec.verify(tokens)
        logits.append(dec.get_last_logits())
    return {"logits": logits, "c_attn": c_attn, "c_mlp": c_mlp}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    if case["kind"] == "gemv":
        rows, n_in, n_rows, epi = case["rows"], case["n_in"], case["n_rows"], case["epi"]
        out = rows * n_rows * {"plain": 4, "swiglu": 1, "residual": 8}[epi]
        return {"bytes": 2 * n_in * n_rows + rows * n_in * (4 if case["norm"] else 2) + 2 * n_in * case["norm"] + out,
                "flops": 2.0 * rows * n_in * n_rows}
    if case["kind"] == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 2 * (m * k + n * k) + 4 * m * n, "flops": 2.0 * m * n * k}
    L, d, f, V, S = case["layers"], case["d_model"], case["d_ffn"], case["vocab"], case["prompt"]
    kv = case["kv_heads"] * case["head_dim"]
    attn_w, mlp_w = 2 * d * d + 2 * kv * d, 3 * d * f  # weights of one attention / MLP sublayer

    def passes(rows, pos, n_attn, n_mlp):  # one pass of `rows` rows on top of `pos` cached positions
        keys = rows * pos + rows * (rows + 1) // 2
        return (2.0 * (n_attn * attn_w + n_mlp * mlp_w + V * d) + 4.0 * kv * n_attn * (pos + rows),
                2.0 * rows * (n_attn * attn_w + n_mlp * mlp_w + V * d) + 4.0 * d * n_attn * keys)

    skip_a, skip_m = (L - int(v.sum()) for v in _mask(case))
    todo = []
    if case["kind"] == "draft":
        todo = [(1, S + i, skip_a, skip_m) for i in range(case["steps"])]
    else:
        todo = []
        for r in range(case.get("rounds", 0)):
            if case["kind"] == "session":
                todo += [(1, S + r + j, skip_a, skip_m) for j in range(case["rows"] - 1)]
            todo.append((case["rows"], S + r, L, L))
    each = [passes(*t) for t in todo]
    b, fl = sum(e[0] for e in each), sum(e[1] for e in each)
    if case["kind"] != "draft":  # the prompt: every weight once, the cache and the embedding rows; the LM head for one row
        b += 2.0 * (L * (attn_w + mlp_w) + V * d) + 4.0 * kv * L * S + 2.0 * S * d
        fl += 2.0 * S * L * (attn_w + mlp_w) + 4.0 * d * L * (S * (S + 1) // 2) + 2.0 * V * d
    return {"bytes": b, "flops": fl}


def tolerance(case):
    if case["kind"] == "gemm":
        return {"rel": 2e-5}  # tensor-core sums of up to 11008 exact products: 4.4e-6 from 64 bits at 4096
    if case["kind"] == "gemv":
        if case["epi"] == "swiglu":
            return {"rel": 1e-3}  # flipped bf16 roundings of the output
        return {"rel": 2e-4} if case["norm"] else {"rel": 2e-6}  # flipped bf16 roundings of the normalised input / fp32 sums
    return {"rel": 2e-2}  # bf16 activations and K/V through a few layers


# ---------------------------------------------------------------- 64-bit reference
def _rms(x, gain):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + _EPS) * gain.double()


def _forward(case, w, tokens, pos, allow, drafting):
    """All rows through the decoder in 64 bits. Row i sits at position pos[i], sees the rows allow[i] and, where
    drafting[i], skips the masked sublayers. Returns the final hidden states, per-sublayer cosines [2][L][rows] and
    the rows' K and V per layer."""
    hd, H, G = case["head_dim"], case["heads"], case["kv_heads"]
    half, n = hd // 2, len(tokens)
    inv = torch.exp(-math.log(_THETA) * 2.0 * torch.arange(half, device="cuda", dtype=torch.float64) / hd)
    ang = torch.as_tensor(pos, device="cuda", dtype=torch.float64)[:, None] * inv
    cos, sin = torch.cos(ang)[:, None, :], torch.sin(ang)[:, None, :]

    def rope(t):
        a, b = t[..., :half], t[..., half:]
        return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)

    def close(a, b):
        return (a * b).sum(-1) / (a.norm(dim=-1) * b.norm(dim=-1)).clamp_min(1e-30)

    skip_a, skip_m = _mask(case)
    drafting = torch.as_tensor(drafting, device="cuda")[:, None]
    x = w.embed[torch.as_tensor(tokens, device="cuda").long()].double()
    c_attn, c_mlp, kv = [], [], []
    for l in range(case["layers"]):
        xn = _rms(x, w.attn_norm[l])
        q = rope((xn @ w.wq[l].double().T).view(n, H, hd))
        k = rope((xn @ w.wk[l].double().T).view(n, G, hd))
        v = (xn @ w.wv[l].double().T).view(n, G, hd)
        kv.append((k.reshape(n, -1), v.reshape(n, -1)))
        a = torch.empty(n, H, hd, dtype=torch.float64, device="cuda")
        for h in range(H):
            g = h * G // H
            s = (q[:, h] @ k[:, g].T) / math.sqrt(hd)
            a[:, h] = torch.softmax(s.masked_fill_(~allow, -math.inf), -1) @ v[:, g]
        y = x + a.view(n, -1) @ w.wo[l].double().T
        y = torch.where(drafting, x, y) if skip_a[l] else y
        c_attn.append(close(x, y))
        yn = _rms(y, w.mlp_norm[l])
        t = torch.nn.functional.silu(yn @ w.wg[l].double().T) * (yn @ w.wu[l].double().T)
        z = y + t @ w.wd[l].double().T
        z = torch.where(drafting, y, z) if skip_m[l] else z
        c_mlp.append(close(y, z))
        x = z
    return x, torch.stack(c_attn), torch.stack(c_mlp), kv


def exact(case, seed):
    if case["kind"] == "gemm":
        A, W = _normal((case["m"], case["k"]), seed, 1), _normal((case["n"], case["k"]), seed, 2, _STD)
        return A.double() @ W.double().T
    if case["kind"] == "gemv":
        rows, n_in, n_rows, epi = case["rows"], case["n_in"], case["n_rows"], case["epi"]
        x = _normal((rows, n_in), seed, 2, dtype=torch.float32 if case["norm"] else torch.bfloat16).double()
        if case["norm"]:
            x = _rms(x, _normal((n_in,), seed, 3, _STD, 1.0))
        a = x @ _normal((n_rows, n_in), seed, 1, _STD).double().T
        if epi == "plain":
            return [a]
        if epi == "swiglu":
            return [torch.nn.functional.silu(a[:, 0::2]) * a[:, 1::2]]
        before = _normal((rows, n_rows), seed, 4, dtype=torch.float32).double()
        after = before + a
        return [after, (before * after).sum(-1) / (before.norm(dim=-1) * after.norm(dim=-1))]

    prompt, tokens = _tokens(case, seed)
    S = case["prompt"]
    # rows: the committed ones in order (the prompt, then row 0 of every round), then the branches
    committed = list(prompt) + ([] if case["kind"] in ("prefill", "draft") else list(tokens[:, 0]))
    toks, pos, drafting = list(committed), list(range(len(committed))), [False] * len(committed)
    branches, outputs = [], []  # branch: (first row, rows, committed rows seen); output: the rows of one logits array

    def branch(part, base, draft):
        first = len(toks)
        toks.extend(part)
        pos.extend(range(base, base + len(part)))
        drafting.extend([draft] * len(part))
        branches.append((first, len(part), base))
        return list(range(first, first + len(part)))

    if case["kind"] == "draft":
        outputs = [[r] for r in branch(tokens, S, True)]
    elif case["kind"] != "prefill":
        for r, row in enumerate(tokens):
            if case["kind"] == "session":
                outputs += [[i] for i in branch(row[:-1], S + r, True)]
            outputs.append([S + r] + branch(row[1:], S + r + 1, False))
    n = len(toks)
    allow = torch.zeros(n, n, dtype=torch.bool, device="cuda")
    nc = len(committed)
    allow[:nc, :nc] = torch.ones(nc, nc, dtype=torch.bool, device="cuda").tril_()
    for first, count, seen in branches:
        allow[first:first + count, :seen] = True
        allow[first:first + count, first:first + count] = torch.ones(count, count, dtype=torch.bool, device="cuda").tril_()

    w = _Weights(case, seed)
    x, c_attn, c_mlp, kv = _forward(case, w, toks, pos, allow, drafting)
    similar = {"c_attn": c_attn[:, :S].mean(-1), "c_mlp": c_mlp[:, :S].mean(-1)}

    def logits_of(rows):
        return _rms(x[rows], w.final_norm) @ w.lm_head.double().T

    if case["kind"] == "prefill":
        return {"logits": logits_of([S - 1])[0], **similar, "kv": [torch.stack([k[S - 1], v[S - 1]]) for k, v in kv]}
    out = {"logits": [logits_of(rows) for rows in outputs]}
    return out if case["kind"] == "draft" else {**out, **similar}
