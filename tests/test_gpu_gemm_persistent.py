"""The persistent GEMM's bias + GELU epilogue over many tiles a CTA with a short K,
where its warps run tiles apart: every element against float64, and the same bits
again.  And what it has to share with the kernels that take the other sizes."""
import ctypes as C
import math

import pytest

from paper_2202_11836_gb300 import _lib as L

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def P(t):
    return C.c_void_p(0 if t is None else int(t.data_ptr()))


def bias_gelu(M, N, K, a, w, bias):
    c = torch.full((M, N), -7.0, dtype=torch.bfloat16, device="cuda")
    gp = torch.full((M, N), -7.0, dtype=torch.float16, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    L.call("sky_gemm", L.SKY_GEMM_XWT, M, N, K, L.SKY_DTYPE_BF16, P(a), P(w), P(c), L.SKY_DTYPE_BF16,
           L.SKY_EPI_BIAS_GELU, P(bias), None, P(gp), None, 0, P(st),
           C.c_void_p(int(torch.cuda.current_stream().cuda_stream)))
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    return c, gp


# 27 tiles a pair (every row tile crosses all eight column tiles); 5 a pair with a
# ragged last row and column tile; 3 to 4 a single CTA
@pytest.mark.parametrize("M,N,K", [(65536, 2048, 256), (2000, 10000, 72), (200, 60000, 72)])
def test_bias_of_many_tiles(M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + N)
    a = torch.randn(M, K, device="cuda", generator=g).bfloat16()
    w = (0.05 * torch.randn(N, K, device="cuda", generator=g)).bfloat16()
    # another value in every column, and a step between column tiles
    bias = torch.randn(N, device="cuda", generator=g)
    bias = (bias + (torch.arange(N, device="cuda") // 256 % 5 - 2)).bfloat16()
    c, gp = bias_gelu(M, N, K, a, w, bias)
    for r in range(0, M, 8192):
        z = a[r:r + 8192].double() @ w.double().T + bias.double()
        phi = 0.5 * (1 + torch.erf(z / math.sqrt(2)))
        ref, dref = z * phi, phi + z * torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)
        # half an ulp of the outputs (2^-9 bf16, 2^-11 fp16) and as much for the sums;
        # the erf formula: 2.5e-5, half of it in Phi
        assert bool(((c[r:r + 8192] - ref).abs() <= 2.0 ** -8 * ref.abs() + 2e-5 * (1 + z.abs())).all())
        assert bool(((gp[r:r + 8192] - dref).abs() <= 2.0 ** -10 * dref.abs() + 3e-5).all())
    for _ in range(3):
        c2, gp2 = bias_gelu(M, N, K, a, w, bias)
        assert torch.equal(c, c2) and torch.equal(gp, gp2)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("M,N,K", [(70, 136, 840), (1100, 1152, 2240), (2000, 3000, 72), (200, 20000, 72)])
def test_bias_before_the_gelu_gradient(M, N, K, dtype):
    """A bias given with GELU_BWD is added first, in every kernel."""
    g = torch.Generator(device="cuda").manual_seed(M + N)
    dt, at = (torch.bfloat16, torch.float16) if dtype == "bf16" else (torch.float32, torch.float32)
    a = torch.randn(M, K, device="cuda", generator=g).to(dt)
    w = (0.05 * torch.randn(N, K, device="cuda", generator=g)).to(dt)
    bias = torch.randn(N, device="cuda", generator=g).to(dt)
    aux = (0.5 + 0.3 * torch.randn(M, N, device="cuda", generator=g)).to(at)
    c = torch.full((M, N), -7.0, dtype=dt, device="cuda")
    code = L.SKY_DTYPE_BF16 if dtype == "bf16" else L.SKY_DTYPE_FP32
    L.call("sky_gemm", L.SKY_GEMM_XWT, M, N, K, code, P(a), P(w), P(c), code, L.SKY_EPI_GELU_BWD, P(bias), P(aux),
           None, None, 0, None, C.c_void_p(int(torch.cuda.current_stream().cuda_stream)))
    ref = (a.double() @ w.double().T + bias.double()) * aux.double()
    # an output's rounding (2^-9 at most for bf16); fp32 sums of K terms
    assert float((c - ref).norm() / ref.norm()) <= (4e-3 if dtype == "bf16" else 1e-5)


@pytest.mark.parametrize("M,N", [(64, 256), (300, 8008), (129, 20000)])
def test_gelu_of_infinities(M, N):
    """GELU of an overflowed pre-activation is the same in both kernels (the cluster
    kernel takes the first shape): +inf of +inf, NaN of NaN."""
    K = 64
    g = torch.Generator(device="cuda").manual_seed(N)
    a = torch.randn(M, K, device="cuda", generator=g).bfloat16()
    w = (0.05 * torch.randn(N, K, device="cuda", generator=g)).bfloat16()
    bias = torch.randn(N, device="cuda", generator=g).bfloat16()
    bias[3::17], bias[5::17], bias[7::17] = math.inf, math.nan, 1e30
    c, _ = bias_gelu(M, N, K, a, w, bias)
    z = a.double() @ w.double().T + bias.double()
    ref = z * 0.5 * (1 + torch.erf(z / math.sqrt(2)))
    inf, nan = torch.isinf(ref), torch.isnan(ref)
    assert torch.equal(torch.isnan(c), nan) and bool((c[inf] == math.inf).all())
    f = ~(inf | nan)
    assert bool(((c[f] - ref[f]).abs() <= 2.0 ** -8 * ref[f].abs() + 2e-5 * (1 + z[f].abs())).all())


# both sides of the lines for long K ranges (152 SMs, k-blocks of 64): 36 tiles to 135,
# 12 to 200, 96 to 88, 192 to 88 (their pairs' last wave is a quarter full), 256: none
@pytest.mark.parametrize("M,N,kb", [(384, 768, 135), (384, 768, 136), (128, 768, 200), (128, 768, 201), (768, 1024, 88),
                                    (768, 1024, 89), (1024, 1536, 88), (1024, 1536, 89), (1024, 2048, 89)])
@pytest.mark.parametrize("ragged", [False, True])
def test_long_weight_gradients(M, N, kb, ragged):
    """With a workspace for split sums and without one; each repeats itself."""
    K = 64 * kb - (3 if ragged else 0)
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    a = torch.randn(K, M, device="cuda", generator=g).bfloat16()
    b = (0.05 * torch.randn(K, N, device="cuda", generator=g)).bfloat16()
    ref = a.double().T @ b.double()
    nb = L.lib().sky_gemm_workspace_bytes(L.SKY_GEMM_XTW, M, N, K, L.SKY_DTYPE_BF16, L.SKY_DTYPE_FP32)
    ws = torch.empty(max(16, nb), dtype=torch.uint8, device="cuda")
    for w, n in ((ws, nb), (None, 0), (ws, max(0, nb - 16))):
        outs = []
        for _ in range(2):
            c = torch.full((M, N), -7.0, device="cuda")
            L.call("sky_gemm", L.SKY_GEMM_XTW, M, N, K, L.SKY_DTYPE_BF16, P(a), P(b), P(c), L.SKY_DTYPE_FP32,
                   L.SKY_EPI_STORE, None, None, None, P(w), n, None,
                   C.c_void_p(int(torch.cuda.current_stream().cuda_stream)))
            outs.append(c)
        # fp32 sums of K products of bf16 values
        assert float((outs[0] - ref).norm() / ref.norm()) <= 1e-5
        assert torch.equal(*outs)
