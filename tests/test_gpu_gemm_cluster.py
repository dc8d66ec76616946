"""The cluster GEMM (small tiles, K split over a cluster's CTAs) at the sizes
where it can go wrong: remainders in every dimension, a K range shorter than
its splits' share, both sides of every line of its dispatch, and each epilogue
after a split, against the same products in float64."""
import ctypes as C

import numpy as np
import pytest

from oracle import encoder_f64 as ORC
from paper_2202_11836_gb300 import _lib as L
from paper_2202_11836_gb300 import synth
from paper_2202_11836_gb300.synth import round_bf16
from parity_util import compare_slice, l2rel, oracle_slice, run_gpu_slice, to_device, to_host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def P(t):
    return C.c_void_p(0 if t is None else int(t.data_ptr()))


def run_gemm(form, M, N, K, a, b, out_dtype, epi=L.SKY_EPI_STORE, bias=None, aux=None, aux_out=None):
    """C (with a guard band of 0xA5 behind it, checked) and the status word."""
    n = M * N
    raw = torch.full((n + 64,), -7.0, dtype=out_dtype, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    L.call("sky_gemm", form, M, N, K, L.SKY_DTYPE_BF16, P(a), P(b), P(raw),
           L.SKY_DTYPE_FP32 if out_dtype == torch.float32 else L.SKY_DTYPE_BF16, epi, P(bias), P(aux),
           P(aux_out), None, 0, P(st), C.c_void_p(int(torch.cuda.current_stream().cuda_stream)))
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    assert bool((raw[n:] == -7.0).all()), "wrote past C"
    return raw[:n].view(M, N)


# (M, N, K) in (tiles of 128 x 64, k-blocks of 64): one tile and one k-block; a
# ragged tail everywhere; two, three and six splits with uneven shares (the
# k-blocks do not divide), 19 / 20 and 38 / 39 tiles of them; 76 / 77, 152 / 153
# and 304 / 305 tiles; pairs with two splits and a ragged last row tile;
# 128-wide weight-gradient tiles
SHAPES = [(1, 8, 8), (129, 72, 200), (70, 136, 13 * 64 + 8), (257, 200, 17 * 64), (61, 72, 35 * 64 + 16),
          (40, 19 * 64, 14 * 64), (40, 20 * 64, 14 * 64), (200, 19 * 64, 13 * 64), (200, 20 * 64, 13 * 64),
          (128, 76 * 64, 136), (128, 77 * 64, 24 * 64), (260, 1664, 25 * 64 + 8),
          (128, 152 * 64, 136), (128, 153 * 64, 72), (2 * 128, 152 * 64, 64), (129, 19520, 64),
          (1100, 1152, 35 * 64), (1100, 1152, 41 * 64), (300, 1200, 33 * 64 + 24), (1000, 2496, 72),
          (130, 160, 97 * 64)]


@pytest.mark.parametrize("form", [L.SKY_GEMM_XWT, L.SKY_GEMM_XW, L.SKY_GEMM_XTW])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_products(form, shape):
    M, N, K = shape
    if form == L.SKY_GEMM_XTW:
        M = (M + 7) // 8 * 8  # its contiguous dimension
        K = K - 3 if K > 8 else K  # and a token count that is no multiple of 8
    elif K % 8:
        K = (K + 7) // 8 * 8
    g = np.random.default_rng(M + 3 * N + 5 * K + form)
    A = round_bf16(g.normal(0, 1, (K, M) if form == L.SKY_GEMM_XTW else (M, K)).astype(np.float32))
    B = round_bf16(g.normal(0, 0.05, (N, K) if form == L.SKY_GEMM_XWT else (K, N)).astype(np.float32))
    a, b = to_device(A, "bf16"), to_device(B, "bf16")
    ad, bd = a.double(), b.double()
    ref = {L.SKY_GEMM_XWT: lambda: ad @ bd.T, L.SKY_GEMM_XW: lambda: ad @ bd,
           L.SKY_GEMM_XTW: lambda: ad.T @ bd}[form]().cpu().numpy()
    bias = round_bf16(g.normal(0, 0.5, N).astype(np.float32))
    # fp32 sums of K products of bf16 values: a few ulp of sqrt(K) terms; bf16
    # output: half an ulp, 2^-9
    c = run_gemm(form, M, N, K, a, b, torch.float32)
    assert l2rel(to_host(c), ref) <= 1e-5
    again = run_gemm(form, M, N, K, a, b, torch.float32)
    assert torch.equal(c, again)  # the splits are added in a fixed order
    cb = run_gemm(form, M, N, K, a, b, torch.bfloat16, bias=to_device(bias, "bf16"))
    assert l2rel(to_host(cb), ref + bias) <= 4e-3


@pytest.mark.parametrize("shape", [(70, 136, 13 * 64 + 8), (129, 200, 24 * 64), (61, 72, 35 * 64 + 16),
                                   (1100, 1152, 35 * 64)], ids=lambda s: "x".join(map(str, s)))
def test_epilogues_after_a_split(shape):
    M, N, K = shape
    g = np.random.default_rng(M + N + K)
    A = round_bf16(g.normal(0, 1, (M, K)).astype(np.float32))
    W = round_bf16(g.normal(0, 0.03, (N, K)).astype(np.float32))
    bias = round_bf16(g.normal(0, 0.5, N).astype(np.float32))
    a, w, b = to_device(A, "bf16"), to_device(W, "bf16"), to_device(bias, "bf16")
    acc = (a.double() @ w.double().T).cpu().numpy()
    gp = torch.full((M, N), -7.0, dtype=torch.float16, device="cuda")
    c = run_gemm(L.SKY_GEMM_XWT, M, N, K, a, w, torch.bfloat16, L.SKY_EPI_BIAS_GELU, b, aux_out=gp)
    assert l2rel(to_host(c), ORC.gelu(acc + bias)) <= 4e-3
    assert l2rel(to_host(gp), ORC.gelu_grad(acc + bias)) <= 1e-3
    d = torch.from_numpy(g.normal(0.5, 0.3, (M, N)).astype(np.float32)).cuda().half()
    c = run_gemm(L.SKY_GEMM_XWT, M, N, K, a, w, torch.bfloat16, L.SKY_EPI_GELU_BWD, aux=d)
    assert l2rel(to_host(c), acc * to_host(d)) <= 4e-3


@pytest.mark.parametrize("batch,seq", [(1, 37), (3, 101), (9, 128)])
def test_slice_with_split_products(batch, seq):
    """Residual, LayerNorm-residual and column-sum epilogues after splits of the
    K range (768 and 3072 long at base width), two layers against the oracle."""
    w = synth.custom(f"split-{batch}x{seq}", layers=2, hidden=768, heads=12, ffn=3072, seq=seq, batch=batch,
                     len_lo=max(1, seq // 3), len_hi=seq, dy_std=1e-2)
    params = synth.slice_params(w, affine="random")
    X, lens, dY = synth.activations(w), synth.lengths(w), synth.upstream_grad(w)
    Y, dX, grads = run_gpu_slice(w, X, lens, dY, params, None)
    compare_slice(w, Y, dX, grads, *oracle_slice(w, X, lens, dY, params))


@pytest.mark.parametrize("M,N,K", [(300, 8008, 136), (129, 20000, 72), (1000, 2600, 200)])
@pytest.mark.parametrize("shift", [0, 8])
def test_wide_bias_gelu(M, N, K, shift):
    """The persistent kernel's bias + GELU, whose outputs leave by TMA, with ragged
    rows and columns (pair and single-CTA tiles), and GELU' off the 16-byte grid,
    which the cluster kernel writes."""
    g = np.random.default_rng(M + N)
    A = round_bf16(g.normal(0, 1, (M, K)).astype(np.float32))
    W = round_bf16(g.normal(0, 0.1, (N, K)).astype(np.float32))
    bias = round_bf16(g.normal(0, 0.5, N).astype(np.float32))
    a, w, b = to_device(A, "bf16"), to_device(W, "bf16"), to_device(bias, "bf16")
    pre = (a.double() @ w.double().T).cpu().numpy() + bias
    raw = torch.full((shift // 2 + M * N + 64,), -7.0, dtype=torch.float16, device="cuda")
    gp = raw[shift // 2:shift // 2 + M * N]
    c = run_gemm(L.SKY_GEMM_XWT, M, N, K, a, w, torch.bfloat16, L.SKY_EPI_BIAS_GELU, b, aux_out=gp)
    assert bool((raw[:shift // 2] == -7.0).all()) and bool((raw[shift // 2 + M * N:] == -7.0).all())
    assert l2rel(to_host(c), ORC.gelu(pre)) <= 4e-3
    assert l2rel(to_host(gp).reshape(M, N), ORC.gelu_grad(pre)) <= 1e-3
