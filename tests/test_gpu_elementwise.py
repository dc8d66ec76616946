"""The element-wise passes around their 16-byte groups: remainders, one element,
and pointers off the 16-byte grid (one element at a time), bit for bit."""
import ctypes as C

import pytest

from paper_2202_11836_gb300 import _lib as L

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def P(t):
    return C.c_void_p(int(t.data_ptr()))


def stream():
    return C.c_void_p(int(torch.cuda.current_stream().cuda_stream))


@pytest.mark.parametrize("n", [1, 3, 4, 1023, 4097, 3_000_002])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_add_and_widen(n, shift):
    a, b = torch.randn(n + shift, device="cuda")[shift:], torch.randn(n + shift, device="cuda")[shift:]
    for dt, code in ((torch.float32, L.SKY_DTYPE_FP32), (torch.bfloat16, L.SKY_DTYPE_BF16)):
        raw = torch.full((shift + n + 8,), -7.0, dtype=dt, device="cuda")
        L.call("sky_add_f32", P(a), P(b), n, code, P(raw[shift:]), stream())
        torch.cuda.synchronize()
        assert torch.equal(raw[shift:shift + n], (a + b).to(dt))
        assert bool((raw[:shift] == -7.0).all()) and bool((raw[shift + n:] == -7.0).all())
        x = raw[shift:shift + n]
        wide = torch.full((shift + n + 8,), -7.0, device="cuda")
        L.call("sky_to_f32", P(x), n, code, P(wide[shift:]), stream())
        torch.cuda.synchronize()
        assert torch.equal(wide[shift:shift + n], x.float())
        assert bool((wide[:shift] == -7.0).all()) and bool((wide[shift + n:] == -7.0).all())
    # in place, as the gradient accumulation uses it
    c = a.clone()
    L.call("sky_add_f32", P(c), P(b), n, L.SKY_DTYPE_FP32, P(c), stream())
    torch.cuda.synchronize()
    assert torch.equal(c, a + b)
