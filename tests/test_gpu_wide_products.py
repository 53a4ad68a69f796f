"""Products of few tokens with wide layers: at most 128 rows, and just one round of 128 x 128 tiles or more."""
import gc

import numpy as np
import pytest
import torch

from paper_2511_11641_b200 import binding as B
from paper_2511_11641_b200 import block as BL
from paper_2511_11641_b200 import layers as L

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _rel(got, want):
    return float(np.linalg.norm(got.double().cpu().numpy() - want) / max(np.linalg.norm(want), 1e-30))


@pytest.mark.parametrize("T", [1, 77, 128])
@pytest.mark.parametrize("k", [9472, 9473, 18944, 18945, 19008])
@pytest.mark.parametrize("act", [B.ACT_GELU_ERF, B.ACT_SWIGLU])
@pytest.mark.parametrize("lin", [False, True])
def test_ffn_few_tokens_wide_layer(T, k, act, lin):
    """At most 128 tokens on layers whose 128 x 128 tiles are just one round of the chip's 148 SMs (k = 18944; SwiGLU 9472) and just
    more (128 x 256 tiles).  Bound: bf16 operands, fp32 sums, saved activations rounded to bf16 (2e-2, as in test_gpu_layers)."""
    g = torch.Generator(device=DEV).manual_seed(T)
    sw, d_m, kp = act == B.ACT_SWIGLU, 136, BL.pad8(k, 2)
    mat = lambda r, c, std: (torch.randn(r, c, generator=g, device=DEV) * std).to(torch.bfloat16)
    X = mat(T, d_m, 1.0)
    wmat = lambda rows_shared: mat(k, d_m, 0.1) if rows_shared else mat(d_m, kp, 0.1)
    w1, w2 = wmat(lin), wmat(not lin)
    w1b = wmat(lin) if sw else None
    b1 = mat(1, kp, 0.5)[0] if not sw else None
    buf = L.ffn_buffers(T, d_m, k, act, torch.bfloat16, DEV, transposed=lin)
    B.ecospa_coupled_ffn_fwd(X, act, w1, w2, k, buf["Y"], buf["H"], buf["A"], w1b_c=w1b, Hb=buf.get("Hb"), b1_c=b1, workspace=buf["ws"],
                             w_in_layout=int(lin), w_out_layout=int(not lin))
    B.ecospa_device_status()
    d = lambda w, rows: w.double().t() if rows else w.double()[:, :k]      # d_m x k
    H = X.double() @ d(w1, lin)
    if sw:
        Hb = X.double() @ d(w1b, lin)
        A = H * torch.sigmoid(H) * Hb
    else:
        H = H + b1[:k].double()
        A = torch.nn.functional.gelu(H)
    errs = {"H": _rel(buf["H"][:, :k], H.cpu().numpy()), "A": _rel(buf["A"][:, :k], A.cpu().numpy()),
            "Y": _rel(buf["Y"], (A @ d(w2, not lin).t()).cpu().numpy())}
    if sw:
        errs["Hb"] = _rel(buf["Hb"][:, :k], Hb.cpu().numpy())
    assert max(errs.values()) <= 2e-2, errs


@pytest.mark.parametrize("T,pairs", [(1, False), (128, False), (129, True)])
def test_cta_pairs_need_more_than_128_rows(T, pairs):
    """The second CTA of a pair holds rows 128 to 255 of a tile: a launch without such rows takes single CTAs, however many tiles."""
    n, d_m = 6656, 256
    X, W = torch.zeros(T, d_m, dtype=torch.bfloat16, device=DEV), torch.zeros(d_m, n, dtype=torch.bfloat16, device=DEV)
    out = [torch.zeros(T, n, dtype=torch.bfloat16, device=DEV) for _ in range(3)]
    ws = torch.empty(B.ecospa_proj_workspace_bytes(T, d_m, n, B.BF16) + 16, dtype=torch.uint8, device=DEV)
    call = lambda: B.ecospa_coupled_qkv_fwd(X, W, W, W, n, n, *out, workspace=ws)
    call()
    torch.cuda.synchronize()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if "gemm_kernel" in e.name]
    del prof
    gc.collect()                                              # (the profiler's records refer to one another, and to this frame)
    if not names:
        pytest.skip("no kernel records from the profiler")
    assert [("gemm_kernel<1," in x or "gemm_kernel<true," in x) for x in names] == [pairs], names


@pytest.mark.parametrize("T,d_m,n,slim", [(1, 3072, 768, True), (1, 3136, 768, False), (1, 2048, 4160, True), (1, 2112, 4160, False), (1, 3072, 4096, True),
                                          (31, 4096, 2048, False), (32, 4096, 2048, True), (128, 4096, 504, False), (128, 4096, 512, True), (129, 4096, 256, True)])
def test_narrow_tiles_on_few_rows(T, d_m, n, slim):
    """Which of the two single-CTA tiles a product of few rows takes, on both sides of each line of the rule (48 tiles of 64 columns, 32 on
    contractions above 4096, 128 KB of X, 128 rows), and its values.  Bound: bf16 operands, fp32 sums, the output's rounding."""
    g = torch.Generator(device=DEV).manual_seed(T)
    x, w = torch.randn(T, n, generator=g, device=DEV).bfloat16(), (torch.randn(n, d_m, generator=g, device=DEV) * 0.05).bfloat16()
    out = torch.zeros(T, d_m, dtype=torch.bfloat16, device=DEV)
    B.ecospa_coupled_vo_fwd_o(x, w, n, out)
    B.ecospa_device_status()
    assert _rel(out, (x.double() @ w.double()).cpu().numpy()) <= 4e-3
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        B.ecospa_coupled_vo_fwd_o(x, w, n, out)
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if "gemm_kernel" in e.name]
    del prof
    gc.collect()
    if not names:
        pytest.skip("no kernel records from the profiler")
    assert ["gemm_kernel<3," in s for s in names] == [slim], names
