"""bf16 attention beside values that no result may depend on: keys past a
sequence's valid length, and the other sequences of the batch."""
import ctypes as C

import pytest

from paper_2202_11836_gb300 import _lib as L

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

D = 64


def P(t):
    return C.c_void_p(0 if t is None else int(t.data_ptr()))


def inputs(B, S, A, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    qkv = torch.randn(B, S, 3, A, D, device="cuda", generator=g).bfloat16()
    return qkv, torch.randn(B, S, A * D, device="cuda", generator=g).bfloat16()


def attention(qkv, dctx, lens):
    """ctx, lse and dqkv [B, S, 3, A, D] of one forward and backward."""
    B, S, _, A, _ = qkv.shape
    H = A * D
    st = C.c_void_p(int(torch.cuda.current_stream().cuda_stream))
    ln = torch.tensor(lens, dtype=torch.int32, device="cuda")
    ctx = torch.empty(B, S, H, dtype=torch.bfloat16, device="cuda")
    lse = torch.empty(B, A, S, device="cuda")
    L.call("sky_attention_fwd", P(qkv), P(ln), B, S, H, A, L.SKY_DTYPE_BF16, P(ctx), P(lse), None, st)
    nb = L.lib().sky_attention_bwd_workspace_bytes(B, S, H, A)
    ws, dqkv = torch.empty(nb, dtype=torch.uint8, device="cuda"), torch.empty_like(qkv)
    L.call("sky_attention_bwd", P(qkv), P(ctx), P(dctx), P(lse), P(ln), B, S, H, A, L.SKY_DTYPE_BF16, P(dqkv), P(ws),
           nb, None, st)
    torch.cuda.synchronize()
    return ctx, lse, dqkv


@pytest.mark.parametrize("S,lens", [(200, [150, 64]), (129, [129, 1]), (384, [128, 300]), (128, [65, 100]), (37, [9, 37])])
def test_scores_of_padded_keys_may_overflow(S, lens):
    A = 2
    qkv, dctx = inputs(2, S, A, S)
    want = attention(qkv, dctx, lens)
    big = qkv.clone()
    for b, n in enumerate(lens):
        big[b, n:, 1] = 3e38  # their products with the queries overflow
    got = attention(big, dctx, lens)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    for b, n in enumerate(lens):
        assert not got[2][b, n:, 1:].any()  # dK and dV of padded keys: exactly zero
    assert torch.equal(got[2], want[2])


@pytest.mark.parametrize("S", [32, 64, 96, 128, 192])
def test_other_sequences_may_be_nan(S):
    """Lengths of whole 32-row blocks (the forward's step; from 129 tokens on 64-row
    ones): no row of the next sequence meets this one's."""
    A, B = 2, 3
    qkv, dctx = inputs(B, S, A, S)
    lens = [S, S, max(1, S - 5)]
    want = attention(qkv, dctx, lens)
    q2, d2 = qkv.clone(), dctx.clone()
    q2[1], d2[1] = float("nan"), float("inf")
    got = attention(q2, d2, lens)
    for b in (0, 2):
        for g, w in zip(got, want):
            assert torch.equal(g[b], w[b])


@pytest.mark.parametrize("S,n", [(128, 64), (128, 32), (100, 64), (64, 32), (256, 128), (200, 64)])
def test_padded_keys_may_be_nan(S, n):
    """The same for keys past a valid length of whole blocks."""
    A = 2
    qkv, dctx = inputs(2, S, A, S + n)
    want = attention(qkv, dctx, [n, n])
    nan = qkv.clone()
    nan[:, n:, 1:] = float("nan")
    if S % 64:  # the last sequence only: its rows meet no other's queries
        nan[0] = qkv[0]
    for g, w in zip(attention(nan, dctx, [n, n]), want):
        assert torch.equal(g, w)
