"""The forms of the tensor-core attention forward (one or two score buffers, the keys
of a query block over one, two or four CTAs) on both sides of the lines between them,
with lengths that leave splits without keys, against float64."""
import ctypes as C

import numpy as np
import pytest

from paper_2202_11836_gb300 import _lib as L
from parity_util import l2rel, maxrel

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

D = 64


def P(t):
    return C.c_void_p(int(t.data_ptr()))


def forward(qkv, lens, B, S, A):
    """(ctx, lse); nothing behind either is written."""
    n, st = B * S * A * D, C.c_void_p(int(torch.cuda.current_stream().cuda_stream))
    ctx = torch.full((n + 64,), -7.0, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B * A * S + 64,), -7.0, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    L.call("sky_attention_fwd", P(qkv), P(lens), B, S, A * D, A, L.SKY_DTYPE_BF16, P(ctx), P(lse), P(status), st)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and bool((ctx[n:] == -7.0).all()) and bool((lse[B * A * S:] == -7.0).all())
    return ctx[:n].view(B, S, A * D), lse[:B * A * S].view(B, A, S)


@pytest.mark.parametrize("S,A,lens,scale", [
    (129, 3, [129, 1], 1.0), (700, 1, [65], 1.0), (705, 1, [705], 1.0),     # 11 key tiles: one CTA; 12: four
    (769, 2, [769, 64, 65], 3.0), (1000, 2, [1000, 129], 1.0),
    (1472, 7, [1472], 1.0), (1473, 7, [1, 1473], 1.0), (1500, 12, [1437], 3.0),  # 23 and 24 tiles; 4, 2 and 1 CTAs
    (2048, 1, [2048, 1, 193], 1.0), (2048, 9, [2048], 3.0), (2048, 10, [2048, 700], 1.0),
    (200, 16, [200, 128, 129] * 4, 1.0), (200, 16, [200, 64, 1, 191, 65] * 3, 1.0),  # 384 and 480 query blocks
])
def test_forward(S, A, lens, scale):
    B = len(lens)
    g = torch.Generator(device="cuda").manual_seed(S + A)
    qkv = (scale * torch.randn(B, S, 3 * A * D, device="cuda", generator=g)).bfloat16()
    ln = torch.tensor(lens, dtype=torch.int32, device="cuda")
    q, k, v = qkv.double().view(B, S, 3, A, D).permute(2, 0, 3, 1, 4)
    s = (q @ k.transpose(-1, -2) / 8.0).masked_fill(
        (torch.arange(S, device="cuda")[None, :] >= ln[:, None])[:, None, None, :], -np.inf)
    ref = (torch.softmax(s, -1) @ v).permute(0, 2, 1, 3).reshape(B, S, A * D)
    ref_lse = (torch.logsumexp(s, -1) / np.log(2.0)).cpu().numpy()
    for _ in range(3):
        ctx, lse = forward(qkv, ln, B, S, A)
        d = ctx.double().cpu().numpy()
        # P and the result rounded to bf16 (2^-9 each), fp32 sums
        assert l2rel(d, ref.cpu().numpy()) <= 5e-3 and maxrel(d, ref.cpu().numpy()) <= 2e-2
        # base-2 scores of up to 2^7: fp32 rounding of a few 2^-24 of them
        assert np.abs(lse.cpu().numpy() - ref_lse).max() <= 2.0 ** -15


def test_scores_of_minus_infinity():
    """A split whose keys' scores are all -inf adds nothing to the others' sum."""
    S, A = 1024, 1
    g = torch.Generator(device="cuda").manual_seed(7)
    qkv = torch.randn(1, S, 3 * D, device="cuda", generator=g).bfloat16()
    qkv[..., 0], qkv[..., D] = 1.0, 0.0
    few = torch.tensor([256], dtype=torch.int32, device="cuda")
    want, want_lse = forward(qkv, few, 1, S, A)
    qkv[:, 256:, D] = -np.inf
    ctx, lse = forward(qkv, torch.tensor([S], dtype=torch.int32, device="cuda"), 1, S, A)
    # the same keys in one split instead of four: fp32 sums in another order
    assert l2rel(ctx.double().cpu().numpy(), want.double().cpu().numpy()) <= 5e-3
    assert float((lse - want_lse).abs().max()) <= 2.0 ** -15
