"""Sizes at the edges of the kernels' forms, against the CPU oracle or plain indexing: segment widths around one warp's and
one block's share, kept lists whose source span is dense, sparse or unaligned, products of one 128 x 128 tile and around the
number of tiles at which CTA pairs take over, fp32 operands with ragged pitches."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2511_11641_b200 import binding as B
from paper_2511_11641_b200 import block as BL
from paper_2511_11641_b200 import layers as L

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 65, 128, 129, 256, 257, 512, 513, 11264, 11265, 23000])
@pytest.mark.parametrize("rope", [B.ROPE_NONE, B.ROPE_HALF])
def test_score_segment_widths(n, rope):
    """Up to 256 indices a warp, above it two blocks, above 11264 in passes; beside a group of another width."""
    if rope and n % 2:
        pytest.skip("rotation pairs need an even width")
    g = torch.Generator().manual_seed(n)
    segs, d_m = 3, 16
    w = {k: torch.randn(d_m, segs * n, generator=g) for k in ("w1", "w2", "g1", "g2")}
    v = {k: torch.randn(d_m, 2 * 40, generator=g) for k in ("w1", "w2", "g1", "g2")}
    dev = lambda t: {k: x.to(DEV) for k, x in t.items()}
    wd, vd = dev(w), dev(v)
    ps = [B.pair(B.PAIR_PLAIN, segs, n, wd["w1"], wd["w2"], 0, 0, g1=wd["g1"], g2=wd["g2"], rope=rope),
          B.pair(B.PAIR_PLAIN, 2, 40, vd["w1"], vd["w2"], 0, 0, g1=vd["g1"], g2=vd["g2"])]
    ups, fis = torch.empty(segs * n + 80, device=DEV), torch.empty(segs + 2, device=DEV)
    raw, only = torch.empty_like(ups), torch.empty_like(ups)
    B.ecospa_score_pairs(ps, 7.0, ups, raw, fis)
    B.ecospa_score_pairs(ps, 7.0, only)                       # without importance: one block per wide segment
    assert torch.equal(ups, only)
    raw_o, ups_o = O.score_pair(w["w1"], w["w2"], 0, 0, segs, n, rope=rope)
    raw_v, ups_v = O.score_pair(v["w1"], v["w2"], 0, 0, 2, 40)
    for got, a, b in ((ups, ups_o, ups_v), (raw, raw_o, raw_v)):
        np.testing.assert_allclose(got.double().cpu().numpy(), np.concatenate([a.ravel(), b.ravel()]), rtol=1e-5, atol=1e-7)
    want = np.concatenate([O.fisher_pair(w["g1"], w["g2"], 0, 0, segs, n, 7.0).ravel(), O.fisher_pair(v["g1"], v["g2"], 0, 0, 2, 40, 7.0).ravel()])
    np.testing.assert_allclose(fis.double().cpu().numpy(), want, rtol=1e-5)


@pytest.mark.parametrize("rep1,rep2", [(2, 1), (3, 1), (4, 1), (5, 2), (8, 1), (1, 9)])
@pytest.mark.parametrize("n", [31, 64, 65, 128, 129, 300])
def test_score_grouped_heads(rep1, rep2, n):
    """Statistics summed over the heads that a segment stacks, four at a time, around the widths of the kernel's forms."""
    g = torch.Generator().manual_seed(rep1 * n)
    segs, d_m = 3, 24
    w1, g1 = (torch.randn(d_m, segs * rep1 * n, generator=g) for _ in range(2))
    w2, g2 = (torch.randn(segs * rep2 * n, d_m, generator=g) for _ in range(2))
    dv = [t.to(DEV) for t in (w1, w2, g1, g2)]
    p = B.pair(B.PAIR_PLAIN, segs, n, dv[0], dv[1], B.SHARED_COLS, B.SHARED_ROWS, g1=dv[2], g2=dv[3], w1_rep=rep1, w2_rep=rep2)
    ups, fis = torch.empty(segs * n, device=DEV), torch.empty(segs, device=DEV)
    B.ecospa_score_pairs([p], 7.0, ups, None, fis)
    c1 = lambda t: (t.double() ** 2).sum(0).view(segs, rep1, n).sum(1)
    c2 = lambda t: (t.double() ** 2).sum(1).view(segs, rep2, n).sum(1)
    raw = (c1(w1) * c2(w2)).sqrt()
    np.testing.assert_allclose(ups.view(segs, n).double().cpu(), raw / raw.norm(dim=1, keepdim=True), rtol=1e-5, atol=1e-7)
    want = 0.5 * (c1(g1).sum(1) / (d_m * rep1 * n) + c2(g2).sum(1) / (d_m * rep2 * n)) / 7.0
    np.testing.assert_allclose(fis.double().cpu(), want, rtol=1e-5)


@pytest.mark.parametrize("n", [1, 2, 32, 33, 64, 65, 128, 129, 256, 257, 511, 513, 1024, 11264, 11265, 23000])
@pytest.mark.parametrize("values", ["normal", "ties", "wide"])
def test_select_segment_widths(n, values):
    """Every count from one to all at the edges of the two forms; few distinct values; values from zero and denormals to inf."""
    r = np.random.default_rng(n)
    ks = sorted({1, min(2, n), n // 2, n - 1, n} - {0})
    u = {"normal": lambda: np.abs(r.standard_normal(n)), "ties": lambda: r.integers(0, 4, n) * 0.25,
         "wide": lambda: np.where(r.random(n) < 0.1, r.choice([0.0, np.inf, 1e-42, 3e38], n), 10.0 ** r.uniform(-30, 30, n))}[values]
    ups = np.concatenate([u() for _ in ks]).astype(np.float32)
    kept, offs = torch.empty(sum(ks), dtype=torch.int32, device=DEV), torch.empty(len(ks) + 1, dtype=torch.int32, device=DEV)
    B.ecospa_select_aligned_topk(torch.from_numpy(ups).to(DEV), [len(ks)], [n], ks, kept, offs)
    assert np.array_equal(kept.cpu().numpy(), O.select_topk(ups, len(ks), n, ks))
    assert np.array_equal(offs.cpu().numpy(), np.concatenate([[0], np.cumsum(ks)]))


@pytest.mark.parametrize("n", [2, 64, 256, 258, 512, 1024, 11264, 11266, 23000])
@pytest.mark.parametrize("rope", [B.ROPE_NONE, B.ROPE_HALF, B.ROPE_INTERLEAVED])
def test_select_equal_scores(n, rope):
    """Segments whose scores are all the same (zero: what an all-zero matrix scores): the lowest units stay, whatever the count."""
    ks = sorted({2, n // 4 * 2, n - 2, n} - {0})
    segs = [(v, k) for v in (0.0, 0.5) for k in ks]
    ups = torch.cat([torch.full((n,), v) for v, _ in segs]).to(DEV)
    kept = torch.full((sum(k for _, k in segs),), -7, dtype=torch.int32, device=DEV)
    B.ecospa_select_rotation_pairs(ups, [len(segs)], [n], [k for _, k in segs], [rope], kept)
    want = [list(range(k // 2)) + list(range(n // 2, n // 2 + k // 2)) if rope == B.ROPE_HALF else list(range(k)) for _, k in segs]
    assert np.array_equal(kept.cpu().numpy(), np.concatenate([s * n + np.array(w) for s, w in enumerate(want)]))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("every,n_kept", [(1, 255), (1, 3000), (2, 256), (2, 1500), (5, 257), (9, 300), (40, 75), (1, 1)])
@pytest.mark.parametrize("shift", [0, 1])
def test_gather_spans(dtype, every, n_kept, shift):
    """Shared-cols tensors: spans of 256 outputs that are staged four, two or one row ahead, or too wide to be; "no index"
    entries; an input that does not start on a 16-byte boundary; row counts around a tile's."""
    r = np.random.default_rng(every * 1000 + n_kept)
    D = 3000
    idx = np.sort(r.choice(np.arange(0, D, every), n_kept, replace=False)).astype(np.int32)
    idx[r.random(n_kept) < 0.02] = -1
    kept = torch.from_numpy(idx).to(DEV)
    jobs, outs, ins = [], [], []
    for rows in (1, 15, 17, 130):
        t = torch.randn(rows + 1, D + 8, device=DEV).to(dtype)[:rows, shift:shift + D]
        o = torch.full((rows, BL.pad8(n_kept, t.element_size())), 7.0, dtype=dtype, device=DEV)
        jobs.append(B.gather(t, o, B.SHARED_COLS, kept, n_kept, D))
        ins.append(t)
        outs.append(o)
    B.ecospa_compact_tensors(jobs)
    at = torch.from_numpy(np.maximum(idx, 0)).long().to(DEV)
    for t, o in zip(ins, outs):
        want = torch.where(kept[None, :] >= 0, t[:, at], torch.zeros((), dtype=dtype, device=DEV))
        assert torch.equal(o[:, :n_kept], want) and not o[:, n_kept:].any()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("layout", [B.SHARED_COLS, B.SHARED_ROWS])
@pytest.mark.parametrize("n", [37000, 37889, 75777, 76000, 151600, 303200])
def test_gather_tile_heights(dtype, layout, n):
    """Row counts on both sides of those at which a tile takes twice as many rows (8 to 32 kept rows of a shared-rows tensor, 16 to
    128 rows of a shared-cols one), with a small odd job beside the large one in the same launch."""
    r = np.random.default_rng(n)
    jobs, pairs = [], []
    for rows, width, keep in ((n, 24, 17), (13, 11, 7)):
        if layout == B.SHARED_COLS:
            t, idx = torch.randn(rows, width, device=DEV).to(dtype), np.sort(r.choice(width, keep, replace=False))
            o = torch.full((rows, BL.pad8(keep, t.element_size())), 7.0, dtype=dtype, device=DEV)
        else:
            t, idx = torch.randn(rows + 50, width, device=DEV).to(dtype), np.sort(r.choice(rows + 50, rows, replace=False))
            o = torch.full((rows, width), 7.0, dtype=dtype, device=DEV)
        kept = torch.from_numpy(idx.astype(np.int32)).to(DEV)
        jobs.append(B.gather(t, o, layout, kept, len(idx), t.shape[1] if layout == B.SHARED_COLS else t.shape[0]))
        pairs.append((o[:, :keep] if layout == B.SHARED_COLS else o, t[:, kept.long()] if layout == B.SHARED_COLS else t[kept.long()]))
    B.ecospa_compact_tensors(jobs)
    for got, want in pairs:
        assert torch.equal(got, want)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("layout", [B.SHARED_COLS, B.SHARED_ROWS])
@pytest.mark.parametrize("shift", [0, 1])
def test_gather_of_what_the_call_before_gathered(dtype, layout, shift):
    """Calls follow one another without a gap, each reading what the one before has just written into the same buffers, at several
    densities (staged, element by element, unaligned): the third result is the first input at the composed indices."""
    r = np.random.default_rng(5)
    D, other, n1, n2 = 2400, 130, 2000, 150
    lists = [np.sort(r.choice(D, n1, replace=False)), np.sort(r.choice(n1, n2, replace=False)), np.sort(r.choice(n2, 100, replace=False))]
    kept = [torch.from_numpy(i.astype(np.int32)).to(DEV) for i in lists]
    sizes = [D, n1, n2, 100]
    mk = lambda n: (torch.zeros(other, n + 8, dtype=dtype, device=DEV)[:, shift:shift + n] if layout == B.SHARED_COLS
                    else torch.zeros(n, other + 8, dtype=dtype, device=DEV)[:, shift:shift + other])
    bufs = [mk(n) for n in sizes]
    jobs = [[B.gather(bufs[i], bufs[i + 1], layout, kept[i], sizes[i + 1], sizes[i])] for i in range(3)]
    at = torch.from_numpy(lists[0][lists[1]][lists[2]]).to(DEV)
    inputs = [torch.randn(bufs[0].shape, device=DEV).to(dtype) for _ in range(12)]
    got = []
    for x in inputs:
        bufs[0].copy_(x)
        for j in jobs:
            B.ecospa_compact_tensors(j)
        got.append(bufs[3].clone())
    for x, y in zip(inputs, got):
        assert torch.equal(y, x[:, at] if layout == B.SHARED_COLS else x[at])


def test_threshold_counts_of_scores_just_written():
    """Scores and the variable-count selection without a call between them, on changing weights in the same buffers."""
    g = torch.Generator().manual_seed(3)
    n, d_m = 3000, 64
    w = [torch.empty(d_m, n, device=DEV) for _ in range(2)]
    ups, kept, k_out = torch.empty(n, device=DEV), torch.empty(n, dtype=torch.int32, device=DEV), torch.empty(1, dtype=torch.int32, device=DEV)
    ps = [B.pair(B.PAIR_PLAIN, 1, n, w[0], w[1], 0, 0)]
    ws = torch.empty(B.ecospa_score_workspace_bytes(ps), dtype=torch.uint8, device=DEV)
    inputs = [[(torch.randn(d_m, n, generator=g) * torch.exp(s * torch.randn(n, generator=g))).to(DEV) for _ in w] for s in (0.1, 1.0, 0.4, 2.0) * 3]
    got = []
    for x in inputs:
        for a, b in zip(w, x):
            a.copy_(b)
        B.ecospa_score_pairs(ps, 1.0, ups, workspace=ws)
        B.ecospa_select_aligned_threshold(ups, [1], [n], 0.9, kept, k_out, l1=True)
        got.append((ups.clone(), k_out.clone()))
    for u, k in got:
        assert int(k) == int(O.threshold_counts(u.cpu().numpy(), 1, n, 0.9, l1=True)[0])
    assert len({int(k) for _, k in got}) > 4


def _rel(got, want):
    return float(np.linalg.norm(got.double().cpu().numpy() - want) / max(np.linalg.norm(want), 1e-30))


@pytest.mark.parametrize("T,d_m,k", [(1, 64, 40), (33, 64, 1), (127, 72, 31), (128, 128, 64), (129, 136, 65), (300, 264, 129), (1100, 512, 1032), (1664, 1536, 1408)])
@pytest.mark.parametrize("act", [B.ACT_GELU_ERF, B.ACT_SWIGLU])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("lin", [False, True])
def test_ffn_tiles(T, d_m, k, act, dtype, lin):
    """Forward and backward of products from less than one 128 x 128 tile to more tiles than SMs (where the launch changes from
    single CTAs to pairs); the fp32 operands also come with a pitch that is not a multiple of four.  Bound: bf16 operands,
    fp32 sums, saved activations rounded to bf16 (2e-2, as in test_gpu_layers).  (An output of one or two numbers has no such
    bound: a single sum of n rounded products is off by up to 2^-8 of the sum of their magnitudes, sqrt(n) times its own size or
    more, so the smallest cases have one token or one hidden index, not both.)"""
    g = torch.Generator(device=DEV).manual_seed(T)
    sw = act == B.ACT_SWIGLU
    odd = 1 if dtype == torch.float32 else 0
    mat = lambda r, c, pitch, std: (torch.randn(r, pitch, generator=g, device=DEV) * std).to(dtype)[:, :c]
    X, dY = mat(T, d_m, d_m + 2 * odd, 1.0), mat(T, d_m, d_m + 3 * odd, 1.0)
    kp = BL.pad8(k, 2)
    wmat = lambda rows_shared: mat(k, d_m, d_m + odd, 0.1) if rows_shared else mat(d_m, kp, kp + odd, 0.1)
    w1, w2 = wmat(lin), wmat(not lin)
    w1b = wmat(lin) if sw else None
    buf = L.ffn_buffers(T, d_m, k, act, dtype, DEV, transposed=lin)
    lay = {"w_in_layout": int(lin), "w_out_layout": int(not lin)}
    L.ffn_fwd_bwd(X, dY, act, w1, w2, k, buf, w1bc=w1b, bias_grads=not sw, **lay)
    B.ecospa_device_status()
    d = lambda w, rows: w.double().t() if rows else w.double()[:, :k]      # d_m x k
    W1, W2, x, dy = d(w1, lin), d(w2, not lin), X.double(), dY.double()
    H, dA = x @ W1, dy @ W2
    if sw:
        Hb, s = x @ d(w1b, lin), torch.sigmoid(H)
        A, dH, dHb = H * s * Hb, dA * Hb * s * (1 + H * (1 - s)), dA * H * s
        dX = dH @ W1.t() + dHb @ d(w1b, lin).t()
    else:
        A = torch.nn.functional.gelu(H)
        dH = dA * (0.5 * (1 + torch.erf(H / 2 ** 0.5)) + H * torch.exp(-0.5 * H * H) / (2 * np.pi) ** 0.5)
        dX = dH @ W1.t()
    st = lambda gw, rows: (gw.t() if rows else gw).cpu().numpy()
    cut = lambda t, rows: t if rows else t[:, :k]
    errs = {"Y": _rel(buf["Y"], (A @ W2.t()).cpu().numpy()), "dX": _rel(buf["dX"], dX.cpu().numpy()),
            "dW1": _rel(cut(buf["dW1"], lin), st(x.t() @ dH, lin)), "dW2": _rel(cut(buf["dW2"], not lin), st(dy.t() @ A, not lin))}
    if sw:
        errs["dW1b"] = _rel(cut(buf["dW1b"], lin), st(x.t() @ dHb, lin))
    else:
        errs["db1"], errs["db2"] = _rel(buf["db1"], dH.sum(0).cpu().numpy()), _rel(buf["db2"], dy.sum(0).cpu().numpy())
    assert max(errs.values()) <= 2e-2, errs


@pytest.mark.parametrize("batch,seq,heads,w,causal", [(60, 48, 32, 32, False), (60, 48, 32, 64, True), (40, 130, 32, 16, True),
                                                      (40, 130, 32, 48, True), (24, 64, 16, 32, False), (75, 65, 8, 64, False)])
def test_attention_many_short_items(batch, seq, heads, w, causal):
    """More work items per CTA than Q buffers, all or the last of them without a visible key for some of the streams."""
    g = torch.Generator(device=DEV).manual_seed(seq)
    T, off = batch * seq, [w * h for h in range(heads)]
    q, k, v, do = (torch.randn(T, heads * w, generator=g, device=DEV).to(torch.bfloat16) for _ in range(4))
    ctx, dq, dk, dv = (torch.zeros_like(q) for _ in range(4))
    lse = torch.zeros(heads * T, device=DEV)
    ws = torch.empty(B.ecospa_attn_workspace_bytes(batch, seq, heads), dtype=torch.uint8, device=DEV)
    hd = B.heads(off, [w] * heads, off, [w] * heads)
    B.ecospa_coupled_attn_fwd(q, k, v, batch, seq, hd, w ** -0.5, causal, ctx, lse)
    B.ecospa_coupled_attn_bwd(q, k, v, ctx, do, lse, batch, seq, hd, w ** -0.5, causal, dq, dk, dv, ws)
    B.ecospa_device_status()
    split = lambda t: t.double().view(batch, seq, heads, w).transpose(1, 2)
    Q, K, V, D = map(split, (q, k, v, do))
    z = Q @ K.transpose(2, 3) * w ** -0.5
    if causal:
        z = z.masked_fill(torch.ones(seq, seq, device=DEV, dtype=torch.bool).triu(1), -float("inf"))
    want_lse = torch.logsumexp(z, 3)
    p = torch.exp(z - want_lse[..., None])
    C = p @ V
    ds = p * (D @ V.transpose(2, 3) - (D * C).sum(3, keepdim=True)) * w ** -0.5
    assert (lse.view(heads, batch, seq).transpose(0, 1).double() - want_lse).abs().max() <= 2e-3
    for got, want in ((ctx, C), (dq, ds @ K), (dk, ds.transpose(2, 3) @ Q), (dv, p.transpose(2, 3) @ D)):
        err = (split(got) - want).flatten(2).norm(dim=2) / want.flatten(2).norm(dim=2)
        assert float(err.max()) <= 2e-2


@pytest.mark.parametrize("batch,seq,heads,w,causal", [(25, 130, 8, 16, True), (25, 192, 8, 32, True), (25, 160, 8, 32, False), (25, 256, 8, 32, True),
                                                      (40, 257, 32, 16, True), (40, 257, 32, 32, False), (40, 300, 32, 32, True), (40, 384, 16, 16, True)])
def test_attention_many_short_stream_items(batch, seq, heads, w, causal):
    """The same in the forward kernel of key streams: blocks that walk three or more items, of one slice per stream each (up to 192
    positions) or the last several of them without a visible key for the third stream (above 256 positions, causal)."""
    test_attention_many_short_items(batch, seq, heads, w, causal)


@pytest.mark.parametrize("batch,seq,heads,w,causal", [(60, 48, 32, 96, False), (60, 48, 32, 128, True), (40, 130, 32, 96, True), (40, 130, 32, 128, False),
                                                      (75, 65, 8, 112, False)])
def test_attention_many_short_wide_items(batch, seq, heads, w, causal):
    """The same on heads of two column blocks."""
    test_attention_many_short_items(batch, seq, heads, w, causal)
