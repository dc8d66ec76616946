"""sky_gemm refuses bf16 epilogue operands off the 8-byte grid on the host: the
kernels access them in groups of four 16-bit values."""
import ctypes as C

import pytest

from paper_2202_11836_gb300 import _lib as L

torch = pytest.importorskip("torch")


@pytest.mark.skipif(torch.cuda.is_available(), reason="the addresses are made up: host checks only")
@pytest.mark.parametrize("M,N,K", [(64, 128, 128), (8192, 4096, 128)])
@pytest.mark.parametrize("off", [2, 4, 6])
@pytest.mark.parametrize("epi,which", [(L.SKY_EPI_STORE, "bias"), (L.SKY_EPI_BIAS_GELU, "bias"),
                                       (L.SKY_EPI_BIAS_GELU, "aux_out"), (L.SKY_EPI_GELU_BWD, "aux")])
def test_refused(epi, which, off, M, N, K):
    at = {n: 0x100000 * (i + 1) for i, n in enumerate(["A", "B", "C", "bias", "aux", "aux_out"])}
    at[which] += off
    if epi == L.SKY_EPI_GELU_BWD:
        at["bias"] = None
    p = {n: C.c_void_p(a) for n, a in at.items()}
    with pytest.raises(L.SkyError) as e:
        L.call("sky_gemm", L.SKY_GEMM_XWT, M, N, K, L.SKY_DTYPE_BF16, p["A"], p["B"], p["C"], L.SKY_DTYPE_BF16,
               epi, p["bias"], p["aux"], p["aux_out"], None, 0, None, None)
    assert e.value.status == L.SKY_ERR_UNSUPPORTED
