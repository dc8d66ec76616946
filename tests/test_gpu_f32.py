"""The fp32 path's GEMM and attention at the sizes where they can go wrong:
remainders of the 64 x 64 x 32 tiles, odd leading dimensions (scalar loads),
both sides of the K-split's lines, head dims off the 16-byte grid, sequences
around the 16-row and 64-column tiles; against float64."""
import ctypes as C

import numpy as np
import pytest

from paper_2202_11836_gb300 import _lib as L
from parity_util import l2rel, maxrel, to_host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F32 = L.SKY_DTYPE_FP32


def P(t):
    return C.c_void_p(0 if t is None else int(t.data_ptr()))


def stream():
    return C.c_void_p(int(torch.cuda.current_stream().cuda_stream))


# (1, 1, 1): all remainder; 33 / 65 / 130: past a slab, a tile; (5, 7, 1000): eight
# splits of a ragged K; (2624, 640, 256) and (2688, 640, 256): 410 and 420 tiles, either
# side of the last split (eleven CTAs an SM, 152 SMs); (63, 640, 96): three slabs
@pytest.mark.parametrize("form", [L.SKY_GEMM_XWT, L.SKY_GEMM_XW, L.SKY_GEMM_XTW])
@pytest.mark.parametrize("shape", [(1, 1, 1), (65, 33, 130), (5, 7, 1000), (128, 384, 128), (63, 640, 96),
                                   (404, 768, 516), (2432, 640, 256), (2496, 640, 256), (2624, 640, 256),
                                   (2688, 640, 256), (130, 65, 33)],
                         ids=lambda s: "x".join(map(str, s)))
def test_gemm(form, shape):
    M, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn((K, M) if form == L.SKY_GEMM_XTW else (M, K), device="cuda", generator=g)
    B = torch.randn((N, K) if form == L.SKY_GEMM_XWT else (K, N), device="cuda", generator=g)
    bias = torch.randn(N, device="cuda", generator=g)
    ad, bd = A.double(), B.double()
    ref = {L.SKY_GEMM_XWT: lambda: ad @ bd.T, L.SKY_GEMM_XW: lambda: ad @ bd, L.SKY_GEMM_XTW: lambda: ad.T @ bd}[form]()
    outs = []
    for _ in range(2):
        raw = torch.full((M * N + 64,), -7.0, device="cuda")
        L.call("sky_gemm", form, M, N, K, F32, P(A), P(B), P(raw), F32, L.SKY_EPI_STORE, P(bias), None, None, None, 0,
               None, stream())
        torch.cuda.synchronize()
        assert bool((raw[M * N:] == -7.0).all())
        outs.append(raw[:M * N].view(M, N))
    # a sequential fp32 sum of K products: error growing as sqrt(K) ulp
    assert l2rel(to_host(outs[0]), (ref + bias.double()).cpu().numpy()) <= 6e-8 * (2 + K ** 0.5)
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("B,S,A,D,lens", [(1, 1, 1, 64, [1]), (2, 15, 3, 32, [15, 1]), (2, 17, 2, 20, [16, 17]),
                                          (1, 65, 2, 128, [64]), (3, 130, 1, 100, [130, 65, 63]),
                                          (2, 64, 5, 3, [64, 9]), (1, 200, 4, 64, [129]), (2, 70, 3, 33, [70, 2]),
                                          (1, 129, 2, 65, [129])])
def test_attention(B, S, A, D, lens):
    H = A * D
    g = torch.Generator(device="cuda").manual_seed(S + D)
    qkv = torch.randn(B, S, 3 * H, device="cuda", generator=g)
    dctx = torch.randn(B, S, H, device="cuda", generator=g)
    ln = torch.tensor(lens, dtype=torch.int32, device="cuda")
    z = qkv.double().requires_grad_()
    q, k, v = z.view(B, S, 3, A, D).permute(2, 0, 3, 1, 4)
    s = q @ k.transpose(-1, -2) / D ** 0.5
    s = s.masked_fill((torch.arange(S, device="cuda")[None, :] >= ln[:, None])[:, None, None, :], -np.inf)
    ref = (torch.softmax(s, -1) @ v).permute(0, 2, 1, 3).reshape(B, S, H)
    ref_lse = torch.logsumexp(s, -1).detach() / np.log(2.0)
    ref_d = torch.autograd.grad(ref, z, dctx.double())[0]
    ctx, lse = torch.full((B * S * H + 32,), -7.0, device="cuda"), torch.empty(B, A, S, device="cuda")
    L.call("sky_attention_fwd", P(qkv), P(ln), B, S, H, A, F32, P(ctx), P(lse), None, stream())
    dq = torch.full((B * S * 3 * H + 32,), -7.0, device="cuda")
    nb = L.lib().sky_attention_bwd_workspace_bytes(B, S, H, A)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    L.call("sky_attention_bwd", P(qkv), P(ctx), P(dctx), P(lse), P(ln), B, S, H, A, F32, P(dq), P(ws), nb, None, stream())
    torch.cuda.synchronize()
    assert bool((ctx[B * S * H:] == -7.0).all()) and bool((dq[B * S * 3 * H:] == -7.0).all())
    # fp32 dot products of D and S terms, expf at 2 ulp
    c, d = ctx[:B * S * H].view(B, S, H), dq[:B * S * 3 * H].view(B, S, 3 * H)
    assert l2rel(to_host(c), ref.detach().cpu().numpy()) <= 2e-6
    assert maxrel(to_host(lse), ref_lse.cpu().numpy()) <= 2e-6
    assert l2rel(to_host(d), ref_d.cpu().numpy()) <= 3e-6
    for i, n in enumerate(lens):  # padded keys: exactly zero
        assert not d[i, n:, H:].any()


@pytest.mark.parametrize("S,len_,hidden", [(130, 130, 64), (130, 129, 128), (64, 40, 20), (200, 200, 1)])
def test_attention_first_scores_overflow(S, len_, hidden):
    """Keys whose scores overflow to -inf get probability 0, also where they fill the
    first tiles of 64 keys; a row that sees only such keys is NaN, as 0 / 0 is."""
    A, D = 2, 32
    H = A * D
    g = torch.Generator(device="cuda").manual_seed(S + hidden)
    qkv = torch.randn(2, S, 3 * H, device="cuda", generator=g)
    z = qkv.view(2, S, 3, A, D)
    z[:, :, 0, :, 0] = 1e20
    z[:, :, 1, :, 0] = 0.0
    z[:, :hidden, 1, 0, 0] = -1e20  # head 0's first keys, both sequences
    z[1, :, 1, 1, 0] = -1e20        # head 1 of sequence 1: every key
    ln = torch.tensor([len_, len_], dtype=torch.int32, device="cuda")
    ctx, lse = torch.empty(2, S, H, device="cuda"), torch.empty(2, A, S, device="cuda")
    L.call("sky_attention_fwd", P(qkv), P(ln), 2, S, H, A, F32, P(ctx), P(lse), None, stream())
    torch.cuda.synchronize()
    q, k, v = qkv.double().view(2, S, 3, A, D).permute(2, 0, 3, 1, 4)
    s = q[..., 1:] @ k[..., 1:].transpose(-1, -2) / D ** 0.5
    s = s.masked_fill((torch.arange(S, device="cuda") >= len_)[None, None, None, :], -np.inf)
    s[:, 0, :, :hidden] = -np.inf
    ref = (torch.softmax(s, -1) @ v).permute(0, 2, 1, 3)
    ref_lse = torch.logsumexp(s, -1) / np.log(2.0)
    c = ctx.view(2, S, A, D)
    for b, a in ((0, 0), (0, 1), (1, 0)):
        assert l2rel(to_host(c[b, :, a]), ref[b, :, a].cpu().numpy()) <= 2e-6
        assert maxrel(to_host(lse[b, a]), ref_lse[b, a].cpu().numpy()) <= 2e-6
    assert bool(torch.isnan(c[1, :, 1]).all())


@pytest.mark.parametrize("B,S,A,D,lens", [(3, 16, 2, 128, [16, 1, 9]), (2, 8, 3, 64, [8, 5]), (2, 16, 1, 100, [16, 15]),
                                          (1, 3, 2, 32, [2]), (2, 16, 2, 7, [4, 16]), (2, 17, 1, 128, [17, 16])])
def test_attention_of_tiny_sequences(B, S, A, D, lens):
    """Both sides of the backward's narrow tiles."""
    test_attention(B, S, A, D, lens)
