"""What this library's users run, as cases to time and to check.

A user of the encoder-slice library does one of these:

- ``step``: a device's training step over its slice of layers, forward and
  backward, as a replayed CUDA graph or as two direct calls, and takes the
  gradients out (they keep their own optimizer or reduce over replicas);
- ``train``: the same step with the library's own AdamW update behind it;
- ``stage``: one stage of a micro-batched pipeline: M forwards into M stash
  slots, then M backwards that add up the gradients, fp32 at the boundaries;
- ``forward``: the forward pass alone (evaluation, a short batch);
- ``attention_fwd``, ``attention_bwd``, ``ffn_fwd``, ``ffn_bwd``,
  ``layernorm``: a layer's blocks, put together from the kernel-level calls.

Widths, lengths and batches are those of the library's own workloads (base
width 768 x 12 heads, large width 1024 x 16 heads, sequences of 128, 512 and
2048 tokens with ragged valid lengths, the 2-layer fp32 slice of width 128) and
values around them.  ``draw`` spreads over the same ranges.

Values are the workloads' own distributions: activations N(0, 1), weights
N(0, 0.02), gamma around 1, small biases, upstream gradients N(0, dy_std),
valid lengths uniform in [len_lo, S].
"""
import ctypes
import math

import torch

from paper_2202_11836_gb300 import _lib as L
from paper_2202_11836_gb300.slice import EncoderSlice
from paper_2202_11836_gb300.synth import PARAM_NAMES

EPS = 1e-12
HEAD_DIM = 64  # of every bf16 attention
ADAMW = dict(lr=2e-4, beta1=0.9, beta2=0.999, eps=1e-6, weight_decay=0.01)


# ------------------------------------------------------------------- the cases
def listed():
    return [
        # The 2-layer fp32 slice of width 128: the tight-tolerance configuration,
        # and the smallest step, where launches and latency are all there is.
        dict(name="step_tiny_fp32", kind="step", dtype="fp32", layers=2, width=128, heads=2, ffn=512,
             batch=4, seq=32, len_lo=16, dy_std=1e-2, graph=False, io_fp32=False),
        # Evaluating two short sentences through a few base-width layers: direct
        # calls, a handful of rows, weights read from memory once.
        dict(name="forward_short", kind="forward", dtype="bf16", layers=2, width=768, heads=12,
             ffn=3072, batch=2, seq=37, len_lo=9, io_fp32=False),
        # One base-width layer (the smallest slice of the 160-layer model that the
        # allocator hands out), direct calls, with the library's AdamW update.
        dict(name="train_base_adamw", kind="train", dtype="bf16", layers=1, width=768, heads=12,
             ffn=3072, batch=16, seq=128, len_lo=64, dy_std=1e-3, graph=False, io_fp32=False),
        # The base-width workload: 4 layers, 32 sequences of 128, a replayed graph.
        dict(name="step_base_s128", kind="step", dtype="bf16", layers=4, width=768, heads=12, ffn=3072,
             batch=32, seq=128, len_lo=64, dy_std=1e-3, graph=True, io_fp32=False),
        # The benchmark workload: 8 large-width layers, 16 sequences of 512.
        dict(name="step_large_s512", kind="step", dtype="bf16", layers=8, width=1024, heads=16, ffn=4096,
             batch=16, seq=512, len_lo=256, dy_std=1e-3, graph=True, io_fp32=True),
        # A pipeline stage of three base-width layers, 4 micro-batches of 8
        # sequences, fp32 hand-offs and accumulated gradients.
        dict(name="stage_microbatches", kind="stage", dtype="bf16", layers=3, width=768, heads=12,
             ffn=3072, batch=8, seq=128, len_lo=64, dy_std=1e-3, micro=4, io_fp32=True),
        # An fp32 base-width layer on a small odd batch: checking a slice at full
        # precision.
        dict(name="step_fp32_base", kind="step", dtype="fp32", layers=1, width=768, heads=12, ffn=3072,
             batch=4, seq=101, len_lo=50, dy_std=1e-2, graph=False, io_fp32=False),
        # Long-sequence attention of the large width, forward.
        dict(name="attention_fwd_s2048", kind="attention_fwd", dtype="bf16", heads=16, batch=4, seq=2048,
             len_lo=512),
        # Attention backward at an odd length, base width.
        dict(name="attention_bwd_s197", kind="attention_bwd", dtype="bf16", heads=12, batch=24, seq=197,
             len_lo=60),
        # The feed-forward block of the large width, forward: FFN1 + bias + GELU,
        # FFN2 + bias, residual + LayerNorm; an odd number of rows.
        dict(name="ffn_fwd_large", kind="ffn_fwd", dtype="bf16", rows=4999, width=1024, ffn=4096),
        # Its backward at base width: LayerNorm, both data gradients, both weight
        # gradients and the bias gradient.
        dict(name="ffn_bwd_base", kind="ffn_bwd", dtype="bf16", rows=3000, width=768, ffn=3072),
        # Residual + LayerNorm, forward and backward, of a large batch.
        dict(name="layernorm_large", kind="layernorm", dtype="bf16", rows=16384, width=1024),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "train", "stage", "forward", "step_fp32", "attention_fwd",
                       "attention_bwd", "ffn_fwd", "ffn_bwd", "layernorm"])
    if kind in ("step", "train", "stage", "forward"):
        heads = rng.choice([4, 8, 12, 16])
        seq = _log_int(rng, 16, 1024)
        rows = _log_int(rng, max(seq, 64), 8192 if kind != "stage" else 2048)
        c = dict(kind=kind, dtype="bf16", layers=rng.randint(1, 4), width=64 * heads, heads=heads,
                 ffn=256 * heads, batch=max(1, rows // seq), seq=seq, len_lo=rng.randint(1, seq),
                 io_fp32=kind == "stage" or rng.random() < 0.3)
        if kind != "forward":
            c["dy_std"] = 1e-3
        if kind in ("step", "train"):
            c["graph"] = rng.random() < 0.5
        if kind == "stage":
            c["micro"] = rng.randint(2, 4)
        return c
    if kind == "step_fp32":
        dim = rng.choice([32, 64, 128])
        heads = _log_int(rng, 1, 768 // dim)
        seq = _log_int(rng, 8, 256)
        rows = _log_int(rng, seq, 1024)
        return dict(kind="step", dtype="fp32", layers=rng.randint(1, 2), width=dim * heads, heads=heads,
                    ffn=4 * dim * heads, batch=max(1, rows // seq), seq=seq, len_lo=rng.randint(1, seq),
                    dy_std=1e-2, graph=rng.random() < 0.5, io_fp32=False)
    if kind.startswith("attention"):
        seq = _log_int(rng, 8, 2048)
        rows = _log_int(rng, max(seq, 64), 8192)
        return dict(kind=kind, dtype="bf16", heads=rng.randint(2, 16), batch=max(1, rows // seq), seq=seq,
                    len_lo=rng.randint(1, seq))
    rows = _log_int(rng, 16, 8192)
    if kind == "layernorm":
        return dict(kind=kind, dtype="bf16", rows=2 * rows, width=8 * _log_int(rng, 16, 256))
    width = 8 * _log_int(rng, 16, 160)
    return dict(kind=kind, dtype="bf16", rows=rows, width=width, ffn=width * rng.choice([2, 3, 4]))


# ------------------------------------------------------------------ the inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _normal(g, shape, std, dtype, mean=0.0):
    return torch.empty(shape, device="cuda", dtype=torch.float32).normal_(mean, std, generator=g).to(dtype)


def _shapes(H, F):
    return {"Wqkv": (3 * H, H), "bqkv": (3 * H,), "Wo": (H, H), "bo": (H,), "gamma1": (H,), "beta1": (H,),
            "W1": (F, H), "b1": (F,), "W2": (H, F), "b2": (H,), "gamma2": (H,), "beta2": (H,)}


def _layer_params(g, H, F, dtype):
    return {n: _normal(g, s, 0.1 if n.startswith("gamma") else 0.02, dtype,
                       1.0 if n.startswith("gamma") else 0.0) for n, s in _shapes(H, F).items()}


def _lengths(g, n, lo, hi):
    return torch.randint(lo, hi + 1, (n,), device="cuda", dtype=torch.int32, generator=g)


def _slice_inputs(case, seed):
    """Parameters per layer, and x, lens, dy of the whole batch (all micro-batches)."""
    g = _generator(seed)
    H, F, S = case["width"], case["ffn"], case["seq"]
    B = case["batch"] * case.get("micro", 1)
    dt = _dtype(case)
    io = torch.float32 if case["io_fp32"] else dt
    params = [_layer_params(g, H, F, dt) for _ in range(case["layers"])]
    x = _normal(g, (B, S, H), 1.0, dt).to(io)
    lens = _lengths(g, B, case["len_lo"], S)
    dy = _normal(g, (B, S, H), case.get("dy_std", 1e-3), dt).to(io)
    return params, x, lens, dy


def _attention_inputs(case, seed):
    g = _generator(seed)
    B, S, H = case["batch"], case["seq"], HEAD_DIM * case["heads"]
    qkv = _normal(g, (B, S, 3 * H), 1.0, torch.bfloat16)
    lens = _lengths(g, B, case["len_lo"], S)
    dctx = _normal(g, (B, S, H), 1e-2, torch.bfloat16)
    return qkv, lens, dctx


def _ffn_inputs(case, seed):
    g = _generator(seed)
    T, H, F, bf = case["rows"], case["width"], case["ffn"], torch.bfloat16
    p = _layer_params(g, H, F, bf)
    x = _normal(g, (T, H), 1.0, bf)
    dy = _normal(g, (T, H), 1e-2, torch.float32)
    return p, x, dy


def _layernorm_inputs(case, seed):
    g = _generator(seed)
    T, H, bf = case["rows"], case["width"], torch.bfloat16
    a = _normal(g, (T, H), 1.0, torch.float32)
    r = _normal(g, (T, H), 1.0, torch.float32)
    gamma, beta = _normal(g, (H,), 0.1, bf, 1.0), _normal(g, (H,), 0.02, bf)
    dy = _normal(g, (T, H), 1e-2, torch.float32)
    return a, r, gamma, beta, dy


def _pointers(tensors):
    return (ctypes.c_void_p * len(tensors))(*[t.data_ptr() for t in tensors])


def _empty(*shape, dtype=torch.float32):
    return torch.empty(shape, device="cuda", dtype=dtype)


def _scratch(nbytes):
    return torch.empty(max(16, int(nbytes)), device="cuda", dtype=torch.uint8)


# --------------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("step", "train", "stage", "forward"):
        params, x, lens, dy = _slice_inputs(case, seed)
        n = case["layers"]
        sl = EncoderSlice(case["width"], case["heads"], case["ffn"], 0, n, case["batch"], case["seq"],
                          case["dtype"], EPS, io_fp32=case["io_fp32"], stash_slots=case.get("micro", 1))
        torch.cuda.synchronize()
        for i, p in enumerate(params):
            L.call("sky_slice_set_params", sl.h, i, _pointers([p[k] for k in PARAM_NAMES]), 1)
        y, dx = torch.empty_like(x), torch.empty_like(x)
        # the tensors the step's results are copied to, one layer after another
        got = {k: _empty(n, *shape, dtype=_dtype(case) if kind == "train" else torch.float32)
               for k, shape in _shapes(case["width"], case["ffn"]).items()}
        s.update(slice=sl, x=x, lens=lens, dy=dy, y=y, dx=dx, got=got,
                 got_ptr=[_pointers([got[k][i] for k in PARAM_NAMES]) for i in range(n)])
        if kind == "train":
            sl.optimizer_init("adamw", **ADAMW)
        if case.get("graph"):
            sl.step_graph(x, lens, y, dy, dx)
        if kind == "stage":
            m, b = case["micro"], case["batch"]
            s["parts"] = [tuple(t[i * b:(i + 1) * b] for t in (x, lens, y, dy, dx)) for i in range(m)]
    elif kind in ("attention_fwd", "attention_bwd"):
        qkv, lens, dctx = _attention_inputs(case, seed)
        B, S, A = case["batch"], case["seq"], case["heads"]
        H = HEAD_DIM * A
        s.update(qkv=qkv, lens=lens, ctx=_empty(B, S, H, dtype=torch.bfloat16), lse=_empty(B, A, S))
        if kind == "attention_bwd":
            # the forward's results, which a backward starts from
            _attention_fwd(s)
            s.update(dctx=dctx, dqkv=torch.empty_like(qkv),
                     ws=_scratch(L.lib().sky_attention_bwd_workspace_bytes(B, S, H, A)))
    elif kind in ("ffn_fwd", "ffn_bwd"):
        p, x, dy = _ffn_inputs(case, seed)
        T, H, F, bf = case["rows"], case["width"], case["ffn"], torch.bfloat16
        s.update(p=p, x=x, x32=x.float(), dy=dy, g=_empty(T, F, dtype=bf),
                 gp=_empty(T, F, dtype=torch.float16), u=_empty(T, H), y=_empty(T, H, dtype=bf),
                 mean=_empty(T), rstd=_empty(T))
        if kind == "ffn_bwd":
            _ffn_fwd(s)
            lib = L.lib()
            bf_t, f32_t = L.SKY_DTYPE_BF16, L.SKY_DTYPE_FP32
            need = max(lib.sky_layernorm_bwd_workspace_bytes(T, H), lib.sky_column_sum_workspace_bytes(T, F),
                       lib.sky_gemm_workspace_bytes(L.SKY_GEMM_XTW, H, F, T, bf_t, f32_t),
                       lib.sky_gemm_workspace_bytes(L.SKY_GEMM_XTW, F, H, T, bf_t, f32_t),
                       lib.sky_gemm_workspace_bytes(L.SKY_GEMM_XW, T, H, F, bf_t, f32_t))
            s.update(ws=_scratch(need), du32=_empty(T, H), du=_empty(T, H, dtype=bf), dz=_empty(T, F, dtype=bf),
                     dp=_empty(T, H), dx=_empty(T, H), dW1=_empty(F, H), dW2=_empty(H, F), db1=_empty(F),
                     db2=_empty(H), dgamma=_empty(H), dbeta=_empty(H))
    else:
        a, r, gamma, beta, dy = _layernorm_inputs(case, seed)
        T, H, bf = case["rows"], case["width"], torch.bfloat16
        s.update(a=a, r=r, gamma=gamma, beta=beta, dy=dy, u=_empty(T, H), y=_empty(T, H, dtype=bf),
                 mean=_empty(T), rstd=_empty(T), du32=_empty(T, H), du=_empty(T, H, dtype=bf), dgamma=_empty(H),
                 dbeta=_empty(H), dbias=_empty(H), ws=_scratch(L.lib().sky_layernorm_bwd_workspace_bytes(T, H)))
    return s


# ------------------------------------------------------------------------- run
def _stream():
    return torch.cuda.current_stream().cuda_stream


def _ptr(t):
    return None if t is None else t.data_ptr()


def _gemm(form, M, N, K, A, B, C, epilogue=L.SKY_EPI_STORE, bias=None, aux=None, aux_out=None, ws=None):
    L.call("sky_gemm", form, M, N, K, L.SKY_DTYPE_BF16, _ptr(A), _ptr(B), _ptr(C),
           L.SKY_DTYPE_FP32 if C.dtype == torch.float32 else L.SKY_DTYPE_BF16, epilogue, _ptr(bias), _ptr(aux),
           _ptr(aux_out), _ptr(ws), 0 if ws is None else ws.numel(), None, _stream())


def _attention_fwd(s):
    c = s["case"]
    L.call("sky_attention_fwd", _ptr(s["qkv"]), _ptr(s["lens"]), c["batch"], c["seq"], HEAD_DIM * c["heads"],
           c["heads"], L.SKY_DTYPE_BF16, _ptr(s["ctx"]), _ptr(s["lse"]), None, _stream())


def _attention_bwd(s):
    c = s["case"]
    L.call("sky_attention_bwd", _ptr(s["qkv"]), _ptr(s["ctx"]), _ptr(s["dctx"]), _ptr(s["lse"]), _ptr(s["lens"]),
           c["batch"], c["seq"], HEAD_DIM * c["heads"], c["heads"], L.SKY_DTYPE_BF16, _ptr(s["dqkv"]),
           _ptr(s["ws"]), s["ws"].numel(), None, _stream())


def _ffn_fwd(s):
    c, p = s["case"], s["p"]
    T, H, F = c["rows"], c["width"], c["ffn"]
    _gemm(L.SKY_GEMM_XWT, T, F, H, s["x"], p["W1"], s["g"], L.SKY_EPI_BIAS_GELU, bias=p["b1"], aux_out=s["gp"])
    _gemm(L.SKY_GEMM_XWT, T, H, F, s["g"], p["W2"], s["u"], bias=p["b2"])
    L.call("sky_layernorm_fwd", _ptr(s["u"]), _ptr(s["x32"]), _ptr(p["gamma2"]), _ptr(p["beta2"]), T, H, EPS,
           L.SKY_DTYPE_BF16, _ptr(s["u"]), None, _ptr(s["y"]), _ptr(s["mean"]), _ptr(s["rstd"]), _stream())


def _layernorm_bwd(s, gamma, dbias):
    c = s["case"]
    L.call("sky_layernorm_bwd", _ptr(s["dy"]), L.SKY_DTYPE_FP32, None, _ptr(s["u"]), _ptr(gamma),
           _ptr(s["mean"]), _ptr(s["rstd"]), c["rows"], c["width"], L.SKY_DTYPE_BF16, _ptr(s["du32"]), _ptr(s["du"]),
           _ptr(s["dgamma"]), _ptr(s["dbeta"]), _ptr(dbias), _ptr(s["ws"]), s["ws"].numel(), _stream())


def _ffn_bwd(s):
    c, p, ws = s["case"], s["p"], s["ws"]
    T, H, F = c["rows"], c["width"], c["ffn"]
    _layernorm_bwd(s, p["gamma2"], s["db2"])
    _gemm(L.SKY_GEMM_XTW, H, F, T, s["du"], s["g"], s["dW2"], ws=ws)
    _gemm(L.SKY_GEMM_XW, T, F, H, s["du"], p["W2"], s["dz"], L.SKY_EPI_GELU_BWD, aux=s["gp"])
    L.call("sky_column_sum", _ptr(s["dz"]), T, F, L.SKY_DTYPE_BF16, _ptr(s["db1"]), _ptr(ws), ws.numel(), _stream())
    _gemm(L.SKY_GEMM_XTW, F, H, T, s["dz"], s["x"], s["dW1"], ws=ws)
    _gemm(L.SKY_GEMM_XW, T, H, F, s["dz"], p["W1"], s["dp"], ws=ws)
    L.call("sky_add_f32", _ptr(s["dp"]), _ptr(s["du32"]), T * H, L.SKY_DTYPE_FP32, _ptr(s["dx"]), _stream())


def _take(s, call):
    """The slice's gradients (or updated parameters) into the user's tensors on the device."""
    for i, ptrs in enumerate(s["got_ptr"]):
        L.call(call, s["slice"].h, i, ptrs, 1)
    return s["got"]


def run(state):
    s = state
    kind = s["case"]["kind"]
    if kind == "forward":
        return {"y": s["slice"].forward(s["x"], s["lens"], s["y"])}
    if kind in ("step", "train"):
        sl = s["slice"]
        if s["case"]["graph"]:
            sl.launch_step_graph()
        else:
            sl.forward(s["x"], s["lens"], s["y"])
            sl.backward(s["dy"], s["dx"])
        if kind == "step":
            return {"y": s["y"], "dx": s["dx"], **_take(s, "sky_slice_get_grads")}
        sl.optimizer_step(ADAMW["lr"])
        return {"y": s["y"], "dx": s["dx"], **_take(s, "sky_slice_get_params")}
    if kind == "stage":
        sl = s["slice"]
        for m, (x, lens, y, _, _) in enumerate(s["parts"]):
            sl.forward(x, lens, y, slot=m)
        for m, (_, _, _, dy, dx) in enumerate(s["parts"]):
            sl.backward(dy, dx, slot=m, accumulate=m > 0)
        return {"y": s["y"], "dx": s["dx"], **_take(s, "sky_slice_get_grads")}
    if kind == "attention_fwd":
        _attention_fwd(s)
        return {"ctx": s["ctx"], "lse": s["lse"]}
    if kind == "attention_bwd":
        _attention_bwd(s)
        return {"dqkv": s["dqkv"]}
    if kind == "ffn_fwd":
        _ffn_fwd(s)
        return {k: s[k] for k in ("g", "gp", "u", "y", "mean", "rstd")}
    if kind == "ffn_bwd":
        _ffn_bwd(s)
        return {k: s[k] for k in ("dx", "dz", "dW1", "dW2", "db1", "db2", "dgamma", "dbeta")}
    L.call("sky_layernorm_fwd", _ptr(s["a"]), _ptr(s["r"]), _ptr(s["gamma"]), _ptr(s["beta"]), s["case"]["rows"],
           s["case"]["width"], EPS, L.SKY_DTYPE_BF16, _ptr(s["u"]), None, _ptr(s["y"]), _ptr(s["mean"]),
           _ptr(s["rstd"]), _stream())
    _layernorm_bwd(s, s["gamma"], s["dbias"])
    return {k: s[k] for k in ("u", "y", "mean", "rstd", "du32", "du", "dgamma", "dbeta", "dbias")}


# ------------------------------------------------------------------------ work
def work(case):
    kind = case["kind"]
    e = 2 if case["dtype"] == "bf16" else 4
    if kind in ("step", "train", "stage", "forward"):
        H, F, n, S = case["width"], case["ffn"], case["layers"], case["seq"]
        T = case["batch"] * S * case.get("micro", 1)
        keys = (case["len_lo"] + S) / 2
        flops = n * (2 * T * (4 * H * H + 2 * H * F) + 4 * H * T * keys)
        par = n * (4 * H * H + 2 * H * F + 9 * H + F)
        io = 4 if case["io_fp32"] else e
        if kind == "forward":
            return {"bytes": e * par + 2 * io * T * H, "flops": flops}
        out = 4 * par if kind != "train" else (4 * 6 + e) * par  # gradients, or w, m, v read and written
        return {"bytes": e * par + 4 * io * T * H + out, "flops": 3 * flops}
    if kind in ("attention_fwd", "attention_bwd"):
        B, S, A = case["batch"], case["seq"], case["heads"]
        H, keys = HEAD_DIM * A, (case["len_lo"] + S) / 2
        if kind == "attention_fwd":
            return {"bytes": B * S * (2 * 4 * H + 4 * A), "flops": 4 * H * B * S * keys}
        return {"bytes": B * S * (2 * 8 * H + 4 * A), "flops": 8 * H * B * S * keys}
    T, H = case["rows"], case["width"]
    if kind == "layernorm":  # a, r, dy in; u, y, du32, du out
        return {"bytes": T * H * (4 + 4 + 4 + 4 + 2 + 4 + 2) + 8 * T, "flops": 0}
    F = case["ffn"]
    w = 2 * 2 * H * F
    if kind == "ffn_fwd":  # x, x32 in; g, g', u, y out
        return {"bytes": w + T * (2 * H + 4 * H + 2 * F + 2 * F + 4 * H + 2 * H) + 8 * T, "flops": 4 * T * H * F}
    # dy, u, x, g, g' in; dx, dz, dW1, dW2 out
    return {"bytes": 3 * w + T * (4 * H + 4 * H + 2 * H + 2 * F + 2 * F + 4 * H + 2 * F), "flops": 8 * T * H * F}


def tolerance(case):
    # Largest error against exact() over the listed and drawn cases, times about
    # four.  fp32: sums of up to a few thousand fp32 products.  bf16: matrix
    # operands rounded to bf16, fp32 sums; in a slice the error grows with its
    # depth.
    kind = case["kind"]
    if case["dtype"] == "fp32":
        return {"rel": 4e-6, "max": 1e-4}
    if kind in ("step", "train", "stage", "forward"):
        return {"rel": 1.6e-2, "max": 0.3}
    if kind.startswith(("attention", "ffn")):
        return {"rel": 1e-2, "max": 0.2}
    return {"rel": 7e-3, "max": 3e-2}


# ----------------------------------------------------------------------- exact
def _softmax_attention(q, k, v, lens):
    """q, k, v [B, A, S, D]; also the rows' log-sum-exp in base 2."""
    S = q.shape[2]
    z = (q @ k.transpose(-1, -2)) / math.sqrt(q.shape[-1])
    hidden = torch.arange(S, device=z.device)[None, :] >= lens[:, None]
    z = z.masked_fill(hidden[:, None, None, :], -math.inf)
    return torch.softmax(z, -1) @ v, torch.logsumexp(z, -1) / math.log(2.0)


def _heads(qkv, A):
    B, S, W = qkv.shape
    return qkv.view(B, S, 3, A, W // (3 * A)).permute(2, 0, 3, 1, 4)


def _layernorm(u, gamma, beta):
    mean = u.mean(-1, keepdim=True)
    rstd = 1.0 / torch.sqrt((u - mean).square().mean(-1, keepdim=True) + EPS)
    return gamma * ((u - mean) * rstd) + beta, mean[..., 0], rstd[..., 0]


def _gelu(z):
    return z * 0.5 * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _gelu_prime(z):
    return 0.5 * (1.0 + torch.erf(z / math.sqrt(2.0))) + z * torch.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi)


def _layer(x, p, lens, A):
    B, S, H = x.shape
    q, k, v = _heads(x @ p["Wqkv"].T + p["bqkv"], A)
    ctx = _softmax_attention(q, k, v, lens)[0].permute(0, 2, 1, 3).reshape(B, S, H)
    x1 = _layernorm(ctx @ p["Wo"].T + p["bo"] + x, p["gamma1"], p["beta1"])[0]
    return _layernorm(_gelu(x1 @ p["W1"].T + p["b1"]) @ p["W2"].T + p["b2"] + x1, p["gamma2"], p["beta2"])[0]


def _adamw_first(p, g, decay):
    a = ADAMW
    w = p * (1.0 - (a["lr"] * a["weight_decay"] if decay else 0.0))
    # first step: both bias-corrected moments are the gradient's own
    return w - a["lr"] * g / (g.abs() + a["eps"])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "train", "stage", "forward"):
        params, x, lens, dy = _slice_inputs(case, seed)
        ps = [{k: v.double().requires_grad_(kind != "forward") for k, v in p.items()} for p in params]
        x0 = h = x.double().requires_grad_(kind != "forward")
        for p in ps:
            h = _layer(h, p, lens, case["heads"])
        if kind == "forward":
            return {"y": h}
        flat = [p[k] for p in ps for k in PARAM_NAMES]
        dx, *grads = torch.autograd.grad(h, [x0] + flat, dy.double())
        m = len(PARAM_NAMES)
        got = {k: torch.stack(grads[j::m]) for j, k in enumerate(PARAM_NAMES)}
        if kind == "train":
            got = {k: _adamw_first(torch.stack([p[k].detach() for p in ps]), g, k.startswith("W"))
                   for k, g in got.items()}
        return {"y": h.detach(), "dx": dx, **got}
    if kind in ("attention_fwd", "attention_bwd"):
        qkv, lens, dctx = _attention_inputs(case, seed)
        B, S, A = case["batch"], case["seq"], case["heads"]
        z = qkv.double().requires_grad_(kind == "attention_bwd")
        o, lse = _softmax_attention(*_heads(z, A), lens)
        ctx = o.permute(0, 2, 1, 3).reshape(B, S, HEAD_DIM * A)
        if kind == "attention_fwd":
            return {"ctx": ctx, "lse": lse}
        return {"dqkv": torch.autograd.grad(ctx, z, dctx.double())[0]}
    if kind in ("ffn_fwd", "ffn_bwd"):
        p, x, dy = _ffn_inputs(case, seed)
        p, x, dy = {k: v.double() for k, v in p.items()}, x.double(), dy.double()
        z = x @ p["W1"].T + p["b1"]
        g, gp = _gelu(z), _gelu_prime(z)
        u = g @ p["W2"].T + p["b2"] + x
        y, mean, rstd = _layernorm(u, p["gamma2"], p["beta2"])
        if kind == "ffn_fwd":
            return {"g": g, "gp": gp, "u": u, "y": y, "mean": mean, "rstd": rstd}
        du, dgamma, dbeta = _layernorm_grad(dy, u, p["gamma2"], mean, rstd)
        dz = (du @ p["W2"]) * gp
        return {"dx": dz @ p["W1"] + du, "dz": dz, "dW1": dz.T @ x, "dW2": du.T @ g, "db1": dz.sum(0),
                "db2": du.sum(0), "dgamma": dgamma, "dbeta": dbeta}
    a, r, gamma, beta, dy = (t.double() for t in _layernorm_inputs(case, seed))
    u = a + r
    y, mean, rstd = _layernorm(u, gamma, beta)
    du, dgamma, dbeta = _layernorm_grad(dy, u, gamma, mean, rstd)
    return {"u": u, "y": y, "mean": mean, "rstd": rstd, "du32": du, "du": du, "dgamma": dgamma, "dbeta": dbeta,
            "dbias": du.sum(0)}


def _layernorm_grad(dy, u, gamma, mean, rstd):
    xhat = (u - mean[:, None]) * rstd[:, None]
    g = dy * gamma
    du = rstd[:, None] * (g - g.mean(-1, keepdim=True) - xhat * (g * xhat).mean(-1, keepdim=True))
    return du, (dy * xhat).sum(0), dy.sum(0)
