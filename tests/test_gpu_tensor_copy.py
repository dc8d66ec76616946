"""Layer tensors to and from the caller's device buffers in one launch: aligned
and misaligned destinations, buffers at the end of their allocation, and pointers
the launch must not take (host memory), against the host copies."""
import ctypes as C

import numpy as np
import pytest

from paper_2202_11836_gb300 import _lib as L
from paper_2202_11836_gb300 import synth
from paper_2202_11836_gb300.slice import EncoderSlice

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GUARD = 0x5A


def buffers(sizes, shift):
    """One byte buffer per tensor, `shift` bytes into an allocation that ends 64 bytes behind it."""
    raw = [torch.full((n + shift + 64,), GUARD, dtype=torch.uint8, device="cuda") for n in sizes]
    return raw, (C.c_void_p * 12)(*[r.data_ptr() + shift for r in raw])


@pytest.mark.parametrize("dtype,shift", [("bf16", 0), ("bf16", 2), ("bf16", 4), ("fp32", 0), ("fp32", 4), ("bf16", 1)])
def test_device_copies(dtype, shift):
    H, F, heads = 192, 776, 3
    with EncoderSlice(H, heads, F, 5, 7, 2, 24, dtype) as s:
        host = [synth.layer_params(l, H, F, dtype, affine="random") for l in (5, 6)]
        s.set_params(5, host[0])
        e = 2 if dtype == "bf16" else 4
        n = [int(np.prod(s.shapes()[k])) for k in synth.PARAM_NAMES]
        raw, ptrs = buffers([m * e for m in n], shift)
        L.call("sky_slice_get_params", s.h, 5, ptrs, 1)
        L.call("sky_slice_set_params", s.h, 6, ptrs, 1)  # and in again, as layer 6's
        back = s.get_params(6)
        for k, r, m in zip(synth.PARAM_NAMES, raw, n):
            assert np.array_equal(back[k], host[0][k])
            assert bool((r[:shift] == GUARD).all()) and bool((r[shift + m * e:] == GUARD).all())
        x = torch.randn(2, 24, H, device="cuda").to(torch.bfloat16 if dtype == "bf16" else torch.float32)
        ln = torch.tensor([24, 7], dtype=torch.int32, device="cuda")
        s.forward(x, ln)
        s.backward(x)
        raw, ptrs = buffers([m * 4 for m in n], shift)
        L.call("sky_slice_get_grads", s.h, 5, ptrs, 1)
        ref = s.get_grads(5)
        for k, r, m in zip(synth.PARAM_NAMES, raw, n):
            got = r[shift:shift + 4 * m].cpu().numpy().tobytes()
            assert got == np.ascontiguousarray(ref[k]).tobytes()
            assert bool((r[:shift] == GUARD).all()) and bool((r[shift + m * 4:] == GUARD).all())


def test_null_tensor_is_refused():
    with EncoderSlice(64, 1, 64, 0, 1, 1, 8, "bf16") as s:
        with pytest.raises(L.SkyError) as ei:
            L.call("sky_slice_get_params", s.h, 0, (C.c_void_p * 12)(), 1)
        assert ei.value.status == L.SKY_ERR_INVALID_ARG
