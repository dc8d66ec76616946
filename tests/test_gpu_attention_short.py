"""The one-launch attention backward of sequences up to 128, at the edges of its
128-row tile and of the valid length, and one length past it (the two-kernel
backward), against float64; the bias gradient of dQKV in a slice covers its
column sums."""
import ctypes as C

import numpy as np
import pytest

from paper_2202_11836_gb300 import _lib as L
from paper_2202_11836_gb300 import synth
from parity_util import compare_slice, l2rel, maxrel, oracle_slice, run_gpu_slice, to_host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

D = 64


def P(t):
    return C.c_void_p(int(t.data_ptr()))


@pytest.mark.parametrize("S,lens", [(1, [1, 1, 1]), (7, [7, 1, 3]), (64, [64, 63, 1]), (65, [65, 64, 2]),
                                    (127, [127, 65, 64]), (128, [128, 127, 1]), (129, [129, 128, 65])])
def test_backward(S, lens):
    B, A = len(lens), 3
    H = A * D
    g = torch.Generator(device="cuda").manual_seed(S)
    qkv = torch.randn(B, S, 3 * H, device="cuda", generator=g).bfloat16()
    dctx = torch.randn(B, S, H, device="cuda", generator=g).bfloat16()
    ln = torch.tensor(lens, dtype=torch.int32, device="cuda")
    z = qkv.double().requires_grad_()
    q, k, v = z.view(B, S, 3, A, D).permute(2, 0, 3, 1, 4)
    s = (q @ k.transpose(-1, -2) / 8.0).masked_fill(
        (torch.arange(S, device="cuda")[None, :] >= ln[:, None])[:, None, None, :], -np.inf)
    out = (torch.softmax(s, -1) @ v).permute(0, 2, 1, 3).reshape(B, S, H)
    ref = torch.autograd.grad(out, z, dctx.double())[0].cpu().numpy()
    st = C.c_void_p(int(torch.cuda.current_stream().cuda_stream))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ctx, lse = torch.empty(B, S, H, dtype=torch.bfloat16, device="cuda"), torch.empty(B, A, S, device="cuda")
    L.call("sky_attention_fwd", P(qkv), P(ln), B, S, H, A, L.SKY_DTYPE_BF16, P(ctx), P(lse), P(status), st)
    raw = torch.full((B * S * 3 * H + 64,), -7.0, dtype=torch.bfloat16, device="cuda")
    nb = L.lib().sky_attention_bwd_workspace_bytes(B, S, H, A)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    L.call("sky_attention_bwd", P(qkv), P(ctx), P(dctx), P(lse), P(ln), B, S, H, A, L.SKY_DTYPE_BF16, P(raw), P(ws), nb,
           P(status), st)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and bool((raw[B * S * 3 * H:] == -7.0).all())
    d = to_host(raw[:B * S * 3 * H]).reshape(B, S, 3 * H)
    # P, dS and the result rounded to bf16 (2^-9 each), fp32 sums
    assert l2rel(d, ref) <= 5e-3 and maxrel(d, ref) <= 2e-2, (l2rel(d, ref), maxrel(d, ref))
    for i, n in enumerate(lens):  # padded keys: exactly zero
        assert not d[i, n:, H:].any()


@pytest.mark.parametrize("batch,seq", [(5, 128), (3, 90)])
def test_slice(batch, seq):
    w = synth.custom(f"short-{batch}x{seq}", layers=1, hidden=256, heads=4, ffn=512, seq=seq, batch=batch, len_lo=1,
                     len_hi=seq, dy_std=1e-2)
    params = synth.slice_params(w, affine="random")
    X, lens, dY = synth.activations(w), synth.lengths(w), synth.upstream_grad(w)
    Y, dX, grads = run_gpu_slice(w, X, lens, dY, params, None)
    compare_slice(w, Y, dX, grads, *oracle_slice(w, X, lens, dY, params))
