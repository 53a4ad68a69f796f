"""What this library is timed on: the work that a coupled-sparsity training run has it do.

Every case goes through the entry points that a training program calls (`binding`,
`layers.ffn_fwd_bwd`), on buffers that such a program keeps from one call to the next.  Five kinds of work:

  sparsify   scores and importance of every pair of a model, aligned top-k, padding of the kept lists, compaction of
             weights, gradients and biases: what a run does each time it re-estimates what to keep
  alg1       one pass of the data-dependent form: importance -> pairs -> threshold counts, read back -> removal from
             weights, gradients, moments and biases
  train      forward and backward of one compacted block (projections, attention core, output projection, FFN)
  forward    the forward half alone: evaluation and serving of a compacted model
  attention  the attention core alone, forward and backward, with query heads sharing K/V heads

Shapes are those of `workloads.py` plus generic ones.  Values: weights as a trained model has them (normal entries, each
shared index with a scale of its own, log-normally spread), gradients likewise, activations N(0, 1).
"""
from __future__ import annotations

import math
import random

import torch

from paper_2511_11641_b200 import binding as B
from paper_2511_11641_b200 import block as BL
from paper_2511_11641_b200 import layers as L

DEV = "cuda"


def _case(kind, name=None, **kw):
    c = {"kind": kind, "layers": 1, "heads": 16, "kv_heads": 0, "d_h": 64, "d_ffn": 4096, "ffn": "gelu", "dtype": "bf16",
         "batch": 1, "seq": 1024, "bias": False, "sparsity": 0.5, "ragged": False, "linear": False, "rope": "none",
         "causal": True, "heavy": False}
    assert set(kw) <= set(c), kw
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest call: one fp32 block of 4 heads (the one-block configuration): all launches and host work.
        _case("sparsify", "sparsify_block_f32", heads=4, d_ffn=1024, dtype="f32", batch=4, seq=128, bias=True),
        # A whole 24-layer GELU model with biases (GPT-2-Medium shape), 0.6 GB of weights.
        _case("sparsify", "sparsify_gpt2m", layers=24, batch=8, bias=True),
        # One wide layer (LLaMA-7B shape) with heavy-tailed weights, stored as a framework's linear layers keep them, its
        # Q/K pairs under rotary embedding; three quarters go.
        _case("sparsify", "sparsify_llama7b_layer", heads=32, d_h=128, d_ffn=11008, ffn="swiglu", batch=2, seq=4096,
              sparsity=0.75, linear=True, rope="half", heavy=True),
        # The largest: all 22 layers of a SwiGLU model (LLaMA-1B shape), 4.5 GB of weights and gradients.
        _case("sparsify", "sparsify_llama1b", layers=22, heads=32, d_ffn=5632, ffn="swiglu", batch=4, seq=2048),
        # One data-dependent pass over 12 layers with Adam moments in fp32 and biases (GPT-2-Small shape): 30 % of the pairs
        # lose their weakest tenth of the score mass.
        _case("alg1", "alg1_gpt2s", layers=12, heads=12, d_ffn=3072, batch=8, bias=True, sparsity=0.1),
        # Training step of the small fp32 block: 512 tokens, launch latency.  (The attention core takes bf16 only; an
        # fp32 block's projections and FFN are what the library does for it.)
        _case("train", "train_block_f32", heads=4, d_ffn=1024, dtype="f32", batch=4, seq=128, bias=True),
        # Ragged head widths (20 ... 64 of 64), an odd FFN width and odd sequence length, 2 x 160 tokens (GPT-2-Small).
        _case("train", "train_gpt2s_ragged", heads=12, d_ffn=3072, batch=2, seq=160, bias=True, ragged=True),
        # Ordinary training step of a GELU block with biases, weights as linear layers keep them.
        _case("train", "train_gpt2m", batch=8, bias=True, linear=True),
        # The benchmark's block: SwiGLU, 4 x 2048 tokens, half of the indices kept.
        _case("train", "train_llama1b", heads=32, d_ffn=5632, ffn="swiglu", batch=4, seq=2048),
        # The largest training step: 2 x 4096 tokens, 128-wide heads cut to 96.
        _case("train", "train_llama7b_layer", heads=32, d_h=128, d_ffn=11008, ffn="swiglu", batch=2, seq=4096, sparsity=0.25),
        # Encoder evaluation: 32 sequences of 197 positions, no mask, 6 heads of ragged widths.
        _case("forward", "forward_encoder_197", heads=6, d_ffn=1536, batch=32, seq=197, bias=True, ragged=True, causal=False),
        # Grouped-query attention: 32 query heads on 8 K/V heads, sequences of 1000.
        _case("attention", "attention_gqa", heads=32, kv_heads=8, batch=4, seq=1000, ragged=True, sparsity=0.3),
    ]


def _loguniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# What a drawn case may cost at most (the largest listed cases of the two sorts of bound).
_MAX_FLOPS = 6.0e12
_MAX_BYTES = 6.5e9


def draw(rng: random.Random):
    """One more case of the same ranges: kind, sizes (log-uniform, odd ones too), storage, type and options."""
    while True:
        kind = rng.choice(["sparsify", "sparsify", "alg1", "train", "train", "train", "forward", "attention"])
        d_h = rng.choice([32, 64, 64, 64, 128])
        heads = max(2, min(32, int(round(_loguniform(rng, 4 if d_h > 32 else 8, 32)))))
        d_m = heads * d_h
        d_ffn = int(d_m * rng.uniform(2.0, 4.0))
        if rng.random() < 0.5:
            d_ffn = (d_ffn + 63) // 64 * 64
        elif kind == "alg1" or kind == "sparsify":
            d_ffn = (d_ffn + 7) // 8 * 8
        tokens = _loguniform(rng, 256, 8192)
        seq = int(_loguniform(rng, 48, min(4096, tokens)))
        if rng.random() < 0.5:
            seq = max(32, (seq + 31) // 32 * 32)
        batch = max(1, int(tokens / seq))
        c = _case(kind, heads=heads, d_h=d_h, d_ffn=d_ffn, batch=batch, seq=seq,
                  ffn=rng.choice(["gelu", "gelu_tanh", "swiglu", "swiglu"]), bias=rng.random() < 0.5,
                  sparsity=round(rng.uniform(0.1, 0.8), 3), ragged=rng.random() < 0.4, linear=rng.random() < 0.35,
                  causal=rng.random() < 0.7, heavy=rng.random() < 0.3)
        if c["ffn"] == "swiglu":
            c["bias"] = False
        if kind in ("sparsify", "train", "alg1") and rng.random() < 0.2:
            c["dtype"] = "f32"
        if kind in ("sparsify", "alg1"):
            c["layers"] = int(_loguniform(rng, 1, 24))
            c["rope"] = rng.choice(["none", "none", "half", "interleaved"])
            if kind == "alg1":
                c["sparsity"] = round(rng.uniform(0.03, 0.3), 3)
        if kind == "attention":
            rep = rng.choice([1, 2, 4, 8])
            if heads % rep:
                continue
            c["kv_heads"] = heads // rep if rep > 1 else 0
        w = work(c)
        if w["flops"] <= _MAX_FLOPS and w["bytes"] <= _MAX_BYTES:
            return c


# ---------------------------------------------------------------------------------------------
# sizes
# ---------------------------------------------------------------------------------------------

def _dtype(c):
    return torch.float32 if c["dtype"] == "f32" else torch.bfloat16


def _esize(c):
    return 4 if c["dtype"] == "f32" else 2


def _kept(n, share):
    return max(1, min(n, int(math.floor(share * n + 0.5))))


def _head_counts(c, salt, n=None):
    """Kept indices of every head: the same for all, or spread around the mean as the method leaves them."""
    n = n or c["heads"]
    even = c["rope"] != "none"
    r = random.Random(1000 * c["heads"] + 10 * c["d_h"] + salt)
    out = []
    for _ in range(n):
        share = 1.0 - c["sparsity"]
        if c["ragged"]:
            share = min(1.0, max(0.15, share * r.uniform(0.6, 1.5)))
        k = _kept(c["d_h"], share)
        out.append(max(2, k - k % 2) if even else k)
    return out


def _counts(c):
    return _head_counts(c, 1), _head_counts(c, 2), _kept(c["d_ffn"], 1.0 - c["sparsity"])


def _pairs_visible(c):
    s = c["seq"]
    return c["batch"] * (s * (s + 1) // 2 if c["causal"] else s * s)


def _attn_flops(c, qk, vo, backward):
    per = 2.0 * _pairs_visible(c)
    f = per * (sum(qk) + sum(vo))
    if backward:
        f += per * (3 * sum(qk) + 2 * sum(vo))
    return f


def _act(c):
    return {"gelu": B.ACT_GELU_ERF, "gelu_tanh": B.ACT_GELU_TANH, "swiglu": B.ACT_SWIGLU}[c["ffn"]]


def work(case):
    """One pass: inputs read once, outputs written once; the products' operations with the counts really kept."""
    c = case
    e, d_m, d_ffn = _esize(c), c["heads"] * c["d_h"], c["d_ffn"]
    D, sw = c["heads"] * c["d_h"], c["ffn"] == "swiglu"
    qk, vo, k = _counts(c)
    n_qk, n_vo = sum(qk), sum(vo)
    T = c["batch"] * c["seq"]
    up = 2 if sw else 1
    if c["kind"] == "sparsify":
        dense = 4 * d_m * D + (up + 1) * d_m * d_ffn
        kept = 2 * d_m * (n_qk + n_vo) + (up + 1) * d_m * k
        by = 2.0 * e * c["layers"] * (dense + kept)          # weights and gradients: read once, the kept part written
        return {"bytes": by, "flops": 4.0 * c["layers"] * dense}
    if c["kind"] == "alg1":
        dense = 4 * d_m * D + (up + 1) * d_m * d_ffn
        by = c["layers"] * dense * (2 * e + 8.0) * 1.9       # weights, gradients, two fp32 moments; most of it stays
        return {"bytes": by, "flops": 4.0 * c["layers"] * dense}
    if c["kind"] == "attention":
        kq, kv = _kv_counts(c)
        rep = c["heads"] // len(kq)
        a = T * ((rep + 1) * sum(kq) + sum(kv) + 2 * rep * sum(kv))   # Q, K, V, dCtx in, Ctx out; then dQ, dK, dV out
        return {"bytes": 2.0 * (a + T * ((rep + 1) * sum(kq) + sum(kv))), "flops": _attn_flops(c, kq * rep, kv * rep, True)}
    proj = 2.0 * T * d_m * (2 * n_qk + 2 * n_vo)
    ffn = 2.0 * T * d_m * k * (up + 1)
    weights = d_m * (2 * n_qk + 2 * n_vo) + (up + 1) * d_m * k
    attn = c["dtype"] == "bf16"
    if c["kind"] == "forward":
        by = e * (weights + T * d_m * 3 + T * (2 * n_qk + 2 * n_vo)) + 2.0 * T * k * (up + 1)
        return {"bytes": by, "flops": proj + ffn + _attn_flops(c, qk, vo, False)}
    # training: x, dY, dOut in; Y, Out, dX out; weights in, weight gradients out; the saved tensors written once
    by = e * (2 * weights + T * d_m * 6 + T * (4 * n_qk + 4 * n_vo)) + 2.0 * T * k * (up + 1)
    return {"bytes": by, "flops": 3 * (proj + ffn) + (_attn_flops(c, qk, vo, True) if attn else 0.0)}


def tolerance(case):
    c = case
    if c["kind"] in ("sparsify", "alg1"):
        # scores and importance are sums of fp32 products; kept sets and compacted tensors follow from them exactly
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}
    # bf16 operands with fp32 accumulation, intermediate tensors rounded to bf16 between the calls.  Against the same chain
    # in 64 bits: up to 4.3e-3 (dW_Q, dW_K: four roundings), 2.9e-3 for one call's outputs; single values up to 0.11.
    return {"rel": 1.5e-2 if c["kind"] == "train" else 1e-2, "max": 0.45}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------

class _Gen:
    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(seed)

    def normal(self, shape, std, dtype):
        t = torch.randn(shape, generator=self.g, device=DEV, dtype=torch.float32)
        if std != 1.0:
            t.mul_(std)
        return t.to(dtype)

    def matrix(self, rows, cols, shared_axis, std, dtype, heavy=False):
        """Normal entries; every shared index has a scale of its own (log-normal, 0.3), 5 % of them ten times larger in
        a heavy-tailed matrix."""
        n = cols if shared_axis else rows
        s = torch.exp(0.3 * torch.randn(n, generator=self.g, device=DEV)) * std
        if heavy:
            s = torch.where(torch.rand(n, generator=self.g, device=DEV) < 0.05, 10.0 * s, s)
        t = torch.randn((rows, cols), generator=self.g, device=DEV, dtype=torch.float32)
        t.mul_(s[None, :] if shared_axis else s[:, None])
        return t.to(dtype)


def _names(c):
    """(matrix, its gradient, extent of the shared axis, shared index is the fast axis) of a block."""
    D, lin = c["heads"] * c["d_h"], c["linear"]
    m = [("wq", "gq", D, not lin), ("wk", "gk", D, not lin), ("wv", "gv", D, not lin), ("wo", "go", D, lin),
         ("w1", "g1", c["d_ffn"], not lin)]
    if c["ffn"] == "swiglu":
        m.append(("w1b", "g1b", c["d_ffn"], not lin))
    return m + [("w2", "g2", c["d_ffn"], lin)]


def _dense_model(c, gen):
    """Weights, gradients and biases of all layers, one stacked tensor per kind: a model's parameters in one arena."""
    dt, d_m, Ls = _dtype(c), c["heads"] * c["d_h"], c["layers"]
    t, layout = {}, {}
    for w, g, D, cols in _names(c):
        for nm, std, heavy in ((w, 0.02, c["heavy"]), (g, 1e-3, False)):
            shape = (d_m, D) if cols else (D, d_m)
            t[nm] = torch.empty((Ls,) + shape, dtype=dt, device=DEV)
            for l in range(Ls):
                t[nm][l] = gen.matrix(*shape, 1 if cols else 0, std, dt, heavy)
            layout[nm] = B.SHARED_COLS if cols else B.SHARED_ROWS
    if c["bias"]:
        for nm, D in (("bq", d_m), ("bk", d_m), ("bv", d_m), ("b1", c["d_ffn"])):
            t[nm] = gen.normal((Ls, D), 0.02, dt)
            layout[nm] = B.SHARED_COLS
    return t, layout


_ROPE = {"none": B.ROPE_NONE, "half": B.ROPE_HALF, "interleaved": B.ROPE_INTERLEAVED}


def _prepare_sparsify(c, gen):
    t, layout = _dense_model(c, gen)
    dt, d_m, Ls, H = _dtype(c), c["heads"] * c["d_h"], c["layers"], c["heads"]
    lin, lout = layout["wq"], layout["wo"]
    qk, vo, k = _counts(c)
    pairs, rope = [], []
    for l in range(Ls):
        w = {nm: t[nm][l] for nm in t if nm[0] == "w"}
        g = {nm: t[nm][l] for nm in t if nm[0] == "g"}
        ps = BL.block_pairs(w, H, c["d_h"], c["d_ffn"], g, layout_in=lin, layout_out=lout)
        ps[0].rope = _ROPE[c["rope"]]
        pairs += ps
        rope += [_ROPE[c["rope"]], B.ROPE_NONE, B.ROPE_NONE]
    s = {"kind": "sparsify", "t": t, "pairs": pairs, "rope": rope if c["rope"] != "none" else None,
         "n_seg": [H, H, 1] * Ls, "seg_len": [c["d_h"], c["d_h"], c["d_ffn"]] * Ls, "k": (qk + vo + [k]) * Ls,
         "tokens": float(c["batch"] * c["seq"])}
    s["ups"] = torch.zeros((2 * d_m + c["d_ffn"]) * Ls, dtype=torch.float32, device=DEV)
    s["fisher"] = torch.zeros((2 * H + 1) * Ls, dtype=torch.float32, device=DEV)
    s["kept"] = torch.zeros(sum(s["k"]), dtype=torch.int32, device=DEV)
    s["ws"] = torch.empty(B.ecospa_score_workspace_bytes(pairs), dtype=torch.uint8, device=DEV)
    # heads padded to the 16 columns that the attention kernels want
    (_, qk_w, n_qk), (_, vo_w, n_vo) = BL.padded_head_layout(qk), BL.padded_head_layout(vo)
    src, dst, kk, kp, o_src, o_dst = [], [], [], [], 0, 0
    lists = []
    for l in range(Ls):
        at = o_dst
        for counts, widths in ((qk, qk_w), (vo, vo_w)):
            for n, w_ in zip(counts, widths):
                src.append(o_src); dst.append(o_dst); kk.append(n); kp.append(w_)
                o_src += n; o_dst += w_
        lists.append((at, at + n_qk, o_src))
        o_src += k
    s["pad"] = (src, dst, kk, kp)
    s["kept_p"] = torch.zeros(o_dst, dtype=torch.int32, device=DEV)
    out, jobs = {}, []
    width = {"q": n_qk, "k": n_qk, "v": n_vo, "o": n_vo, "1": k, "2": k}
    for nm in t:
        n = width[nm[1]]
        if t[nm].dim() == 2:
            shape = (Ls, BL.pad8(n, _esize(c)))
        elif layout[nm] == B.SHARED_COLS:
            shape = (Ls, t[nm].shape[1], BL.pad8(n, _esize(c)))
        else:
            shape = (Ls, n, t[nm].shape[2])
        out[nm] = torch.zeros(shape, dtype=dt, device=DEV)
        for l in range(Ls):
            a, b, f = lists[l]
            kept = {"q": s["kept_p"][a:], "k": s["kept_p"][a:], "v": s["kept_p"][b:], "o": s["kept_p"][b:],
                    "1": s["kept"][f:], "2": s["kept"][f:]}[nm[1]]
            jobs.append(B.gather(t[nm][l], out[nm][l], layout[nm], kept[:n], n, c["d_ffn"] if nm[1] in "12" else d_m))
    s["jobs"], s["out"] = jobs, out
    return s


def _run_sparsify(s):
    B.ecospa_score_pairs(s["pairs"], s["tokens"], s["ups"], None, s["fisher"], s["ws"])
    if s["rope"] is None:
        B.ecospa_select_aligned_topk(s["ups"], s["n_seg"], s["seg_len"], s["k"], s["kept"])
    else:
        B.ecospa_select_rotation_pairs(s["ups"], s["n_seg"], s["seg_len"], s["k"], s["rope"], s["kept"])
    B.ecospa_pad_kept(s["kept"], *s["pad"], s["kept_p"])
    B.ecospa_compact_tensors(s["jobs"])
    return {"scores": s["ups"], "importance": s["fisher"], "kept": s["kept"], "out": s["out"]}


def _prepare_alg1(c, gen):
    """Groups of all layers (weights, gradients, Adam moments, biases), a second set of buffers of the same size for what the
    pass leaves, and its workspace: a program that compacts as it trains goes back and forth between two such sets."""
    t, layout = _dense_model(c, gen)
    for nm in [n for n in t if n[0] == "w"]:
        for moment in "mv":
            t[moment + nm[1:]] = torch.rand(t[nm].shape, generator=gen.g, device=DEV)
            layout[moment + nm[1:]] = layout[nm]
    out = {nm: torch.zeros_like(t[nm]) for nm in t}
    lin, lout, H = layout["wq"], layout["wo"], c["heads"]
    sets = []
    for m in (t, out):
        groups = []
        for l in range(c["layers"]):
            w = {nm: m[nm][l] for nm in m}
            aux = lambda names: [(w[nm], layout[nm]) for nm in names if nm in w]
            groups.append(B.group(w["wq"], w["wk"], lin, lin, [c["d_h"]] * H, g1=w["gq"], g2=w["gk"],
                                  aux=aux(["mq", "vq", "mk", "vk", "bq", "bk"]), rope=_ROPE[c["rope"]]))
            groups.append(B.group(w["wv"], w["wo"], lin, lout, [c["d_h"]] * H, g1=w["gv"], g2=w["go"],
                                  aux=aux(["mv", "vv", "mo", "vo", "bv"])))
            groups.append(B.group(w["w1"], w["w2"], lin, lout, [c["d_ffn"]], w1b=w.get("w1b"), g1=w["g1"], g2=w["g2"],
                                  g1b=w.get("g1b"), aux=aux(["m1", "v1", "m1b", "v1b", "m2", "v2", "b1"])))
        sets.append(groups)
    ws = torch.empty(B.ecospa_alg1_workspace_bytes(sets[0]), dtype=torch.uint8, device=DEV)
    at = B.ecospa_alg1_offsets(sets[0])
    view = lambda off, n, dtype: ws[off:off + 4 * n].view(dtype)
    return {"kind": "alg1", "groups": sets[0], "into": sets[1], "out": out, "tokens": float(c["batch"] * c["seq"]), "ws": ws,
            "theta": 1.0 - c["sparsity"], "n_choose": int(0.3 * at[5] + 0.5), "scores": view(at[0], at[4], torch.float32),
            "importance": view(at[1], at[5], torch.float32), "chosen": view(at[2], at[5], torch.int32)}


def _run_alg1(s):
    k = B.ecospa_alg1_plan(s["groups"], s["tokens"], s["n_choose"], s["theta"], True, 2, s["ws"])
    B.ecospa_alg1_apply(s["groups"], k, s["into"], s["ws"])
    return {"scores": s["scores"], "importance": s["importance"], "chosen": s["chosen"], "out": s["out"]}


def _compact_cols(gen, c, d_m, counts, offs, total, std=0.02):
    """A compacted projection weight: `counts` real columns per head in blocks padded with zero columns."""
    cols = BL.pad8(total)
    t = torch.zeros((d_m, cols), dtype=torch.float32, device=DEV)
    for n, o in zip(counts, offs):
        t[:, o:o + n] = torch.randn((d_m, n), generator=gen.g, device=DEV) * std
    return t.to(_dtype(c))


def _prepare_block(c, gen, train):
    """Compacted weights and every buffer of one block, as a training program keeps them."""
    dt, d_m, H = _dtype(c), c["heads"] * c["d_h"], c["heads"]
    T = c["batch"] * c["seq"]
    qk, vo, k = _counts(c)
    (qk_off, qk_w, n_qk), (vo_off, vo_w, n_vo) = BL.padded_head_layout(qk), BL.padded_head_layout(vo)
    lin = c["linear"]
    attn = c["dtype"] == "bf16"
    up = ["w1", "w1b"] if c["ffn"] == "swiglu" else ["w1"]
    w = {"wq": _compact_cols(gen, c, d_m, qk, qk_off, n_qk), "wk": _compact_cols(gen, c, d_m, qk, qk_off, n_qk),
         "wv": _compact_cols(gen, c, d_m, vo, vo_off, n_vo), "wo": _compact_cols(gen, c, d_m, vo, vo_off, n_vo)}
    kp = BL.pad8(k, _esize(c))
    for nm in up + ["w2"]:
        w[nm] = torch.zeros((d_m, kp), dtype=dt, device=DEV)
        w[nm][:, :k] = gen.normal((d_m, k), 0.02, dt)
    real = {"wq": n_qk, "wk": n_qk, "wv": n_vo, "wo": n_vo, "w1": k, "w1b": k, "w2": k}
    rows = {nm for nm in w if (nm in ("wo", "w2")) != lin}        # stored with the shared index as the slow axis
    for nm in rows:
        w[nm] = w[nm].t()[:real[nm]].contiguous()
    if c["bias"]:
        for nm, n in (("bq", n_qk), ("bk", n_qk), ("bv", n_vo), ("b1", k), ("b2", d_m), ("bo", d_m)):
            w[nm] = torch.zeros(BL.pad8(n, _esize(c)), dtype=dt, device=DEV)
            w[nm][:n] = gen.normal((n,), 0.02, dt)
    z = lambda *shape, dtype=dt: torch.zeros(shape, dtype=dtype, device=DEV)
    s = {"kind": "train" if train else "forward", "w": w, "n_qk": n_qk, "n_vo": n_vo, "k": k, "attn": attn,
         "batch": c["batch"], "seq": c["seq"], "causal": c["causal"], "scale": c["d_h"] ** -0.5, "act": _act(c), "bias": c["bias"],
         "lay": {"w_in_layout": B.SHARED_ROWS if lin else B.SHARED_COLS, "w_out_layout": B.SHARED_COLS if lin else B.SHARED_ROWS},
         "heads": B.heads(qk_off, qk_w, vo_off, vo_w)}
    s["x"] = gen.normal((T, d_m), 1.0, dt)
    code = B.BF16 if attn else B.F32
    if attn:
        s["Q"], s["K"], s["V"], s["Ctx"] = z(T, n_qk), z(T, n_qk), z(T, n_vo), z(T, n_vo)
        s["lse"] = z(H * T, dtype=torch.float32)
    else:   # the mixed values and their gradients come from the program's own fp32 attention
        s["Q"], s["K"], s["V"] = z(T, n_qk), z(T, n_qk), z(T, n_vo)
        s["Ctx"] = gen.normal((T, n_vo), 1.0, dt)
    s["Out"] = z(T, d_m)
    s["ffn"] = L.ffn_buffers(T, d_m, k, s["act"], dt, DEV, transposed=lin)
    s["ws"] = torch.empty(B.ecospa_proj_workspace_bytes(T, d_m, max(n_qk, n_vo), code) + 16, dtype=torch.uint8, device=DEV)
    if train:
        s["dY"], s["dOut"] = gen.normal((T, d_m), 1.0, dt), gen.normal((T, d_m), 1.0, dt)
        s["dCtx"] = z(T, n_vo)
        if attn:
            s["dQ"], s["dK"], s["dV"] = z(T, n_qk), z(T, n_qk), z(T, n_vo)
            s["attn_ws"] = torch.empty(B.ecospa_attn_workspace_bytes(c["batch"], c["seq"], H), dtype=torch.uint8, device=DEV)
        else:
            s["dQ"], s["dK"], s["dV"] = gen.normal((T, n_qk), 1.0, dt), gen.normal((T, n_qk), 1.0, dt), gen.normal((T, n_vo), 1.0, dt)
        s["grads"] = {nm: torch.zeros_like(w[nm]) for nm in ("wq", "wk", "wv", "wo")}
        if c["bias"]:
            s["grads"].update({nm: torch.zeros_like(w[nm]) for nm in ("bq", "bk", "bv", "bo")})
    return s


def _forward(s):
    w = s["w"]
    B.ecospa_coupled_qkv_fwd(s["x"], w["wq"], w["wk"], w["wv"], s["n_qk"], s["n_vo"], s["Q"], s["K"], s["V"], bq_c=w.get("bq"),
                             bk_c=w.get("bk"), bv_c=w.get("bv"), workspace=s["ws"], **s["lay"])
    if s["attn"]:
        B.ecospa_coupled_attn_fwd(s["Q"], s["K"], s["V"], s["batch"], s["seq"], s["heads"], s["scale"], s["causal"], s["Ctx"],
                                  s["lse"])
    B.ecospa_coupled_vo_fwd_o(s["Ctx"], w["wo"], s["n_vo"], s["Out"], bo=w.get("bo"), workspace=s["ws"], **s["lay"])


def _run_forward(s):
    w, f = s["w"], s["ffn"]
    _forward(s)
    B.ecospa_coupled_ffn_fwd(s["x"], s["act"], w["w1"], w["w2"], s["k"], f["Y"], f["H"], f["A"], w1b_c=w.get("w1b"),
                             Hb=f.get("Hb"), b1_c=w.get("b1"), b2=w.get("b2"), workspace=f["ws"], **s["lay"])
    return {"Y": f["Y"], "Out": s["Out"], "Ctx": s["Ctx"]}


def _run_train(s):
    w, f, g = s["w"], s["ffn"], s["grads"]
    _forward(s)
    L.ffn_fwd_bwd(s["x"], s["dY"], s["act"], w["w1"], w["w2"], s["k"], f, w1bc=w.get("w1b"), b1c=w.get("b1"), b2=w.get("b2"),
                  bias_grads=s["bias"], **s["lay"])
    B.ecospa_coupled_vo_bwd_o(s["Ctx"], w["wo"], s["n_vo"], s["dOut"], s["dCtx"], g["wo"], g.get("bo"), workspace=s["ws"],
                              **s["lay"])
    if s["attn"]:
        B.ecospa_coupled_attn_bwd(s["Q"], s["K"], s["V"], s["Ctx"], s["dCtx"], s["lse"], s["batch"], s["seq"], s["heads"],
                                  s["scale"], s["causal"], s["dQ"], s["dK"], s["dV"], s["attn_ws"])
    # the block's input gradient: what the FFN left in dX plus the three projections' share
    B.ecospa_coupled_qkv_bwd(s["x"], w["wq"], w["wk"], w["wv"], s["n_qk"], s["n_vo"], s["dQ"], s["dK"], s["dV"], f["dX"], g["wq"],
                             g["wk"], g["wv"], g.get("bq"), g.get("bk"), g.get("bv"), accumulate_dX=True, workspace=s["ws"],
                             **s["lay"])
    out = {"Y": f["Y"], "Out": s["Out"], "dX": f["dX"], "dCtx": s["dCtx"], "dW1": f["dW1"], "dW2": f["dW2"]}
    if "dW1b" in f:
        out["dW1b"] = f["dW1b"]
    elif s["bias"]:
        out["db1"] = f["db1"]
    if s["bias"]:
        out["db2"] = f["db2"]
    if s["attn"]:
        out["Ctx"] = s["Ctx"]
    # the gradient of the K bias under the attention core is zero (a softmax does not see a shift of all its scores): what
    # is computed is rounding noise, which has nothing to compare
    out.update({"d" + nm: v for nm, v in g.items() if not (nm == "bk" and s["attn"])})
    return out


def _kv_counts(c):
    """Kept indices of every K/V head; its query heads share them."""
    n = c["kv_heads"] or c["heads"]
    return _head_counts(c, 1, n), _head_counts(c, 2, n)


def _prepare_attention(c, gen):
    H, T = c["heads"], c["batch"] * c["seq"]
    kq, kv = _kv_counts(c)
    rep = H // len(kq)
    (k_off, _, n_k), (v_off, _, n_v) = BL.padded_head_layout(kq), BL.padded_head_layout(kv)
    hq, hv = [n for n in kq for _ in range(rep)], [n for n in kv for _ in range(rep)]
    (q_off, q_w, n_q), (o_off, o_w, n_o) = BL.padded_head_layout(hq), BL.padded_head_layout(hv)
    hd = B.heads(q_off, q_w, o_off, o_w, k_off, v_off) if rep > 1 else B.heads(q_off, q_w, o_off, o_w)

    def blocks(pitch, counts, offs):
        t = torch.zeros((T, pitch), dtype=torch.bfloat16, device=DEV)
        for n, o in zip(counts, offs):
            t[:, o:o + n] = gen.normal((T, n), 1.0, torch.bfloat16)
        return t
    s = {"kind": "attention", "heads": hd, "batch": c["batch"], "seq": c["seq"], "causal": c["causal"], "scale": c["d_h"] ** -0.5}
    # K and dK share the pitch of Q and dQ, whatever columns they use of it
    s["Q"], s["K"], s["V"], s["dCtx"] = blocks(n_q, hq, q_off), blocks(n_q, kq, k_off), blocks(n_v, kv, v_off), blocks(n_o, hv, o_off)
    for nm, like in (("dQ", "Q"), ("dK", "K"), ("dV", "V"), ("Ctx", "dCtx")):
        s[nm] = torch.zeros_like(s[like])
    s["lse"] = torch.zeros(H * T, dtype=torch.float32, device=DEV)
    s["ws"] = torch.empty(B.ecospa_attn_workspace_bytes(c["batch"], c["seq"], H), dtype=torch.uint8, device=DEV)
    return s


def _run_attention(s):
    B.ecospa_coupled_attn_fwd(s["Q"], s["K"], s["V"], s["batch"], s["seq"], s["heads"], s["scale"], s["causal"], s["Ctx"], s["lse"])
    B.ecospa_coupled_attn_bwd(s["Q"], s["K"], s["V"], s["Ctx"], s["dCtx"], s["lse"], s["batch"], s["seq"], s["heads"], s["scale"],
                              s["causal"], s["dQ"], s["dK"], s["dV"], s["ws"])
    return {"Ctx": s["Ctx"], "lse": s["lse"], "dQ": s["dQ"], "dK": s["dK"], "dV": s["dV"]}


def prepare(case, seed):
    c, gen = case, _Gen(seed)
    if c["kind"] == "sparsify":
        return _prepare_sparsify(c, gen)
    if c["kind"] == "alg1":
        return _prepare_alg1(c, gen)
    if c["kind"] == "attention":
        return _prepare_attention(c, gen)
    return _prepare_block(c, gen, c["kind"] == "train")


_RUN = {"sparsify": _run_sparsify, "alg1": _run_alg1, "train": _run_train, "forward": _run_forward, "attention": _run_attention}


def run(state):
    return _RUN[state["kind"]](state)


# ---------------------------------------------------------------------------------------------
# the same outputs in 64 bits, in plain torch
# ---------------------------------------------------------------------------------------------

def exact(case, seed):
    """What `run` returns, computed in fp64 on the inputs of `prepare`.  Kept lists and what is gathered by them follow the
    fp32 scores (a near-tie may fall either way), so they have no value here."""
    with torch.no_grad():
        if case["kind"] in ("sparsify", "alg1"):
            return _exact_scores(case, seed)
        s = prepare(case, seed)
        if case["kind"] == "attention":
            return _exact_attention(case, s)
        return _exact_block(case, s)


def _exact_scores(c, seed):
    t, _ = _dense_model(c, _Gen(seed))
    sq = lambda x, cols: (x * x).sum(0 if cols else 1)       # over the axis that is not shared
    cols_in, cols_out = not c["linear"], c["linear"]
    up, imp = [], []
    for l in range(c["layers"]):
        x = {nm: t[nm][l] for nm in t}
        for a, b, cols_b, n_seg in (("q", "k", cols_in, c["heads"]), ("v", "o", cols_out, c["heads"]), ("1", "2", cols_out, 1)):
            w1 = x["w" + a].double()
            if a == "1" and "w1b" in x:
                w1 = w1 * x["w1b"].double()
            c1, c2 = sq(w1, cols_in).view(n_seg, -1), sq(x["w" + b].double(), cols_b).view(n_seg, -1)
            n = c1.shape[1]
            rope = c["rope"] if a == "q" else "none"
            if rope == "none":
                raw = c1.sqrt() * c2.sqrt()
                ups = raw / raw.norm(dim=1, keepdim=True)
            else:                                          # the unit is a rotation pair, counted once
                fold = (lambda v: v.view(n_seg, 2, n // 2).sum(1)) if rope == "half" else (lambda v: v.view(n_seg, n // 2, 2).sum(2))
                raw = fold(c1).sqrt() * fold(c2).sqrt()
                u = raw / raw.norm(dim=1, keepdim=True)
                ups = u.repeat(1, 2) if rope == "half" else u.repeat_interleave(2, dim=1)
            mean = lambda nm, cols: sq(x[nm].double(), cols).view(n_seg, -1).sum(1) * n_seg / x[nm].numel()
            m1 = mean("g" + a, cols_in)
            if a == "1" and "g1b" in x:
                m1 = 0.5 * (m1 + mean("g1b", cols_in))
            up.append(ups.reshape(-1))
            imp.append(0.5 * (m1 + mean("g" + b, cols_b)) / (c["batch"] * c["seq"]))
    r = {"scores": torch.cat(up), "importance": torch.cat(imp), "out": None}
    r["kept" if c["kind"] == "sparsify" else "chosen"] = None
    return r


def _blocks16(counts):
    """First column and width of every head's block, widths rounded up to 16."""
    out, at = [], 0
    for n in counts:
        w = -(-n // 16) * 16
        out.append((at, w))
        at += w
    return out


def _exact_core(c, q, k, v, scale, d_ctx=None):
    """softmax(scale q k^T) v of one sequence and head in fp64, its log-sum-exp, and the three gradients."""
    z = scale * (q @ k.t())
    if c["causal"]:
        i = torch.arange(c["seq"], device=z.device)
        z = z.masked_fill(i[None, :] > i[:, None], -math.inf)
    lse = torch.logsumexp(z, 1)
    p = torch.exp(z - lse[:, None])
    ctx = p @ v
    if d_ctx is None:
        return ctx, lse, None
    ds = p * (d_ctx @ v.t() - (d_ctx * ctx).sum(1, keepdim=True)) * scale
    return ctx, lse, (ds @ k, ds.t() @ q, p.t() @ d_ctx)


def _exact_attention(c, s):
    kq, kv = _kv_counts(c)
    rep = c["heads"] // len(kq)
    qb, ob = _blocks16([n for n in kq for _ in range(rep)]), _blocks16([n for n in kv for _ in range(rep)])
    kb, vb = _blocks16(kq), _blocks16(kv)
    S, T = c["seq"], c["batch"] * c["seq"]
    r = {nm: torch.zeros(s[nm].shape, dtype=torch.float64, device=DEV) for nm in ("Ctx", "dQ", "dK", "dV")}
    lse = torch.zeros((c["heads"], T), dtype=torch.float64, device=DEV)
    for b in range(c["batch"]):
        rows = slice(b * S, (b + 1) * S)
        for h in range(c["heads"]):
            cut = lambda blk: slice(blk[0], blk[0] + blk[1])
            q, o, k, v = cut(qb[h]), cut(ob[h]), cut(kb[h // rep]), cut(vb[h // rep])
            ctx, l, (dq, dk, dv) = _exact_core(c, s["Q"][rows, q].double(), s["K"][rows, k].double(), s["V"][rows, v].double(),
                                               s["scale"], s["dCtx"][rows, o].double())
            r["Ctx"][rows, o], lse[h, rows], r["dQ"][rows, q] = ctx, l, dq
            r["dK"][rows, k] += dk
            r["dV"][rows, v] += dv
    r["lse"] = lse.view(-1)
    return r


def _exact_block(c, s):
    train, attn, S = c["kind"] == "train", s["attn"], c["seq"]
    n_qk, n_vo, k, lin = s["n_qk"], s["n_vo"], s["k"], c["linear"]
    w, x = s["w"], s["x"].double()
    real = {"wq": n_qk, "wk": n_qk, "wv": n_vo, "wo": n_vo, "w1": k, "w1b": k, "w2": k}
    rows = {nm for nm in real if (nm in ("wo", "w2")) != lin}   # stored with the shared index as the slow axis
    W = {nm: (w[nm].double().t() if nm in rows else w[nm].double())[:, :real[nm]] for nm in real if nm in w}   # d_m x n
    bias = lambda nm, n: w[nm][:n].double() if nm in w else 0.0
    Q, K, V = x @ W["wq"] + bias("bq", n_qk), x @ W["wk"] + bias("bk", n_qk), x @ W["wv"] + bias("bv", n_vo)
    qk, vo, _ = _counts(c)
    heads = [(slice(a, a + m), slice(e, e + n)) for (a, m), (e, n) in zip(_blocks16(qk), _blocks16(vo))]

    def cores(d_ctx):
        ctx = torch.zeros_like(V)
        g = [torch.zeros_like(Q), torch.zeros_like(K), torch.zeros_like(V)]
        for b in range(c["batch"]):
            r = slice(b * S, (b + 1) * S)
            for i, o in heads:
                ctx[r, o], _, d = _exact_core(c, Q[r, i], K[r, i], V[r, o], s["scale"], None if d_ctx is None else d_ctx[r, o])
                if d is not None:
                    g[0][r, i], g[1][r, i], g[2][r, o] = d
        return ctx, g

    d_ctx = s["dOut"].double() @ W["wo"] if train else None
    if attn:
        ctx, grads = cores(d_ctx)
    else:
        ctx, grads = s["Ctx"].double(), [s[nm].double() for nm in ("dQ", "dK", "dV")] if train else None
    out = {"Out": ctx @ W["wo"].t() + bias("bo", x.shape[1])}
    F = torch.nn.functional
    H = x @ W["w1"] + bias("b1", k)
    if c["ffn"] == "swiglu":
        Hb = x @ W["w1b"]
        sg = torch.sigmoid(H)
        A, dact = H * sg * Hb, None
    else:
        A = F.gelu(H, approximate="tanh" if c["ffn"] == "gelu_tanh" else "none")
    out["Y"] = A @ W["w2"].t() + bias("b2", x.shape[1])
    if attn:
        out["Ctx"] = ctx
    if not train:
        return out
    dY = s["dY"].double()
    dA = dY @ W["w2"]
    if c["ffn"] == "swiglu":
        dH, dHb = dA * Hb * sg * (1 + H * (1 - sg)), dA * H * sg
    elif c["ffn"] == "gelu":
        dH = dA * (0.5 * (1 + torch.erf(H / math.sqrt(2.0))) + H * torch.exp(-0.5 * H * H) / math.sqrt(2.0 * math.pi))
    else:
        t = torch.tanh(math.sqrt(2.0 / math.pi) * (H + 0.044715 * H ** 3))
        dH = dA * (0.5 * (1 + t) + 0.5 * H * (1 - t * t) * math.sqrt(2.0 / math.pi) * (1 + 3 * 0.044715 * H * H))

    def stored(nm, g, like):                                    # d_m x n -> as the weight's gradient is stored
        g = g.t() if nm in rows else g
        r = torch.zeros(like.shape, dtype=torch.float64, device=DEV)
        r[:, :g.shape[1]] = g
        return r

    f, xt = s["ffn"], x.t()
    out.update({"dCtx": d_ctx, "dW1": stored("w1", xt @ dH, f["dW1"]), "dW2": stored("w2", dY.t() @ A, f["dW2"])})
    dX = dH @ W["w1"].t()
    if c["ffn"] == "swiglu":
        out["dW1b"] = stored("w1b", xt @ dHb, f["dW1b"])
        dX += dHb @ W["w1b"].t()
    elif s["bias"]:
        out["db1"] = dH.sum(0)
    for nm, g in zip(("wq", "wk", "wv"), grads):
        dX += g @ W[nm].t()
        out["d" + nm] = stored(nm, xt @ g, s["grads"][nm])
        if s["bias"] and not (nm == "wk" and attn):
            out["db" + nm[1]] = F.pad(g.sum(0), (0, s["grads"]["b" + nm[1]].numel() - g.shape[1]))
    out["dX"] = dX
    out["dwo"] = stored("wo", s["dOut"].double().t() @ ctx, s["grads"]["wo"])
    if s["bias"]:
        out["db2"], out["dbo"] = dY.sum(0), s["dOut"].double().sum(0)
    return out
