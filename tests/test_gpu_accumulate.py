"""Accumulated gradients: the bf16 weight-gradient products and column sums add to
the gradients where they finish, in every tiling and split that products of these
sizes take.  Exact: each adds the number that an overwriting backward stores."""
import numpy as np
import pytest

from paper_2202_11836_gb300 import synth
from paper_2202_11836_gb300.slice import EncoderSlice

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("H,heads,F,B,S,dtype", [
    (64, 1, 72, 1, 1, "bf16"),           # one partial tile, one k-block
    (192, 3, 776, 3, 31, "bf16"),        # partial tiles both ways
    (256, 4, 1024, 16, 64, "bf16"),      # splits of six, three and two
    (768, 12, 3072, 8, 128, "bf16"),     # no split; 64-wide tiles
    (1024, 16, 4096, 3, 500, "bf16"),    # 128-wide tiles
    (768, 12, 3072, 8, 256, "bf16"),     # pair tiles
    (768, 12, 3072, 16, 509, "bf16"),    # partials in the workspace, one remainder block
    (1024, 16, 4096, 16, 512, "bf16"),   # 256-wide tiles
    (192, 3, 776, 3, 31, "fp32"),
])
def test_accumulate(H, heads, F, B, S, dtype):
    g = torch.Generator(device="cuda").manual_seed(H + S)
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    rnd = lambda: torch.randn(B, S, H, device="cuda", generator=g).to(td)
    lens = torch.full((B,), S, dtype=torch.int32, device="cuda")
    lens[0] = (S + 1) // 2
    x, dys = rnd(), [rnd(), rnd(), rnd()]
    with EncoderSlice(H, heads, F, 0, 1, B, S, dtype, stash_slots=2) as s:
        s.set_params(0, synth.layer_params(0, H, F, dtype, affine="random"))

        def grads(dy, accumulate):
            s.backward(dy, accumulate=accumulate)
            s.sync()
            return s.get_grads(0)

        s.forward(x, lens)
        each = [grads(dy, False) for dy in dys]
        want = {k: (each[0][k] + each[1][k]) + each[2][k] for k in each[0]}
        grads(dys[0], False)
        grads(dys[1], True)
        got = grads(dys[2], True)
        for k in want:
            assert np.array_equal(got[k], want[k]), k
