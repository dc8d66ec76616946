"""Failure detection on the GPU without a GPU fault.

A host-side hook makes the GEMM's TMA producer skip its copies; every
consumer wait is time-bounded, so the kernel gives up after the set limit,
reports the timeout in the status word, releases its tensor memory and exits.
The context must stay usable: the same GEMM then runs correctly, and a slice
whose GEMMs timed out reports SKY_ERR_TIMEOUT from sky_slice_sync.
"""
import ctypes as C

import numpy as np
import pytest

from paper_2202_11836_gb300 import _lib as L
from paper_2202_11836_gb300 import synth
from parity_util import l2rel, to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def P(t):
    return C.c_void_p(0 if t is None else int(t.data_ptr()))


def stream():
    return C.c_void_p(int(torch.cuda.current_stream().cuda_stream))


def test_gemm_wait_timeout_is_reported_and_context_survives():
    M, N, K = 256, 512, 256
    g = np.random.default_rng(1)
    A = synth.round_bf16(g.normal(0, 1, (M, K)).astype(np.float32))
    W = synth.round_bf16(g.normal(0, 0.05, (N, K)).astype(np.float32))
    a, w = to_device(A, "bf16"), to_device(W, "bf16")
    c = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    L.lib().sky_debug_gemm_fault(50_000_000, 1)  # 50 ms per wait, no TMA copies
    try:
        L.call("sky_gemm", L.SKY_GEMM_XWT, M, N, K, 0, P(a), P(w), P(c), 0, 0, None, None, None,
               None, 0, P(status), stream())
        torch.cuda.synchronize()
    finally:
        L.lib().sky_debug_gemm_fault(0, 0)
    assert int(status.item()) & 2, "timeout bit not set"
    # the context is intact: the same GEMM now runs and is correct
    status.zero_()
    L.call("sky_gemm", L.SKY_GEMM_XWT, M, N, K, 0, P(a), P(w), P(c), 0, 0, None, None, None,
           None, 0, P(status), stream())
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref = A.astype(np.float64) @ W.astype(np.float64).T
    assert l2rel(c.float().cpu().numpy(), ref) <= 4e-3


def test_slice_reports_timeout_then_recovers():
    from paper_2202_11836_gb300.slice import EncoderSlice
    w = synth.custom("fault", layers=1, hidden=128, heads=2, ffn=256, seq=64, batch=2)
    X, lens = synth.activations(w), synth.lengths(w)
    with EncoderSlice(128, 2, 256, 0, 1, 2, 64) as s:
        s.set_params(0, synth.layer_params(0, 128, 256, "bf16", affine="random"))
        x = to_device(X, "bf16")
        ln = torch.from_numpy(lens).cuda()
        L.lib().sky_debug_gemm_fault(20_000_000, 1)
        try:
            s.forward(x, ln)
            with pytest.raises(L.SkyError) as e:
                s.sync()
            assert e.value.status == L.SKY_ERR_TIMEOUT
        finally:
            L.lib().sky_debug_gemm_fault(0, 0)
        y = s.forward(x, ln)
        s.sync()  # OK again
        assert torch.isfinite(y.float()).all()


# of the persistent kernel: SM pairs and single CTAs, bf16 and fp32 output, each epilogue
@pytest.mark.parametrize("M,N", [(2048, 4096), (200, 25000)])
@pytest.mark.parametrize("epi,f32", [(L.SKY_EPI_STORE, False), (L.SKY_EPI_STORE, True), (L.SKY_EPI_BIAS_GELU, False),
                                     (L.SKY_EPI_GELU_BWD, False)])
def test_persistent_gemm_timeout(M, N, epi, f32):
    """More than two 128 x 64 tiles an SM: the persistent kernel.  Its producer, MMA
    and epilogue warps give up, nothing is stored, and the next call is right."""
    K = 192
    g = torch.Generator(device="cuda").manual_seed(N + epi)
    a = torch.randn(M, K, device="cuda", generator=g).bfloat16()
    w = (0.05 * torch.randn(N, K, device="cuda", generator=g)).bfloat16()
    bias = torch.randn(N, device="cuda", generator=g).bfloat16()
    aux = torch.randn(M, N, device="cuda", generator=g).half()
    out = torch.full((M, N), -7.0, dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    gp = torch.full((M, N), -7.0, dtype=torch.float16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def go():
        L.call("sky_gemm", L.SKY_GEMM_XWT, M, N, K, 0, P(a), P(w), P(out), int(f32), epi, P(bias), P(aux), P(gp), None,
               0, P(status), stream())
        torch.cuda.synchronize()

    L.lib().sky_debug_gemm_fault(20_000_000, 1)
    try:
        go()
    finally:
        L.lib().sky_debug_gemm_fault(0, 0)
    assert int(status.item()) & 2, "timeout bit not set"
    assert bool((out == -7.0).all()) and bool((gp == -7.0).all())
    status.zero_()
    go()
    assert int(status.item()) == 0
    z = a.double() @ w.double().T + bias.double()
    if epi == L.SKY_EPI_BIAS_GELU:
        z = z * 0.5 * (1 + torch.erf(z / 2 ** 0.5))
    elif epi == L.SKY_EPI_GELU_BWD:
        z = z * aux.double()
    assert float((out - z).norm() / z.norm()) <= (1e-5 if f32 else 4e-3)


# of the cluster kernel: unsplit, two, three and six splits, pairs, 128-wide tiles
@pytest.mark.parametrize("form,M,N,K", [(L.SKY_GEMM_XWT, 256, 512, 256), (L.SKY_GEMM_XWT, 700, 768, 1024),
                                        (L.SKY_GEMM_XWT, 384, 768, 1024), (L.SKY_GEMM_XWT, 64, 768, 3072),
                                        (L.SKY_GEMM_XWT, 2048, 768, 3072), (L.SKY_GEMM_XTW, 1024, 4096, 512)])
@pytest.mark.parametrize("skip", [1, 2])
def test_cluster_gemm_timeout_stores_nothing(form, M, N, K, skip):
    """Also where the others' parts of a tile are complete (skip = 2), their sum is
    not stored."""
    g = torch.Generator(device="cuda").manual_seed(M + K)
    a = torch.randn((K, M) if form == L.SKY_GEMM_XTW else (M, K), device="cuda", generator=g).bfloat16()
    w = (0.05 * torch.randn((K, N) if form == L.SKY_GEMM_XTW else (N, K), device="cuda", generator=g)).bfloat16()
    out = torch.full((M, N), -7.0, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def go():
        L.call("sky_gemm", form, M, N, K, 0, P(a), P(w), P(out), 1, 0, None, None, None, None, 0, P(status), stream())
        torch.cuda.synchronize()

    L.lib().sky_debug_gemm_fault(20_000_000, skip)
    try:
        go()
    finally:
        L.lib().sky_debug_gemm_fault(0, 0)
    assert int(status.item()) & 2, "timeout bit not set"
    assert bool((out == -7.0).all())
    status.zero_()
    go()
    assert int(status.item()) == 0
    ref = a.double().T @ w.double() if form == L.SKY_GEMM_XTW else a.double() @ w.double().T
    assert float((out - ref).norm() / ref.norm()) <= 1e-5
