"""The timed cases of the sparse-linear library: what a program that trains, stores, prefills and
decodes with bitmask-compressed linear layers asks of it, through the package's public calls.

Kinds of case (the "op" of a case):
  linear      y = x . (W o Mask)^T for one layer: SparseMatrix.linear with bf16 or INT8 weights,
              from one decode row to a 2048-token prefill.
  w8a8        the same layer with INT8 activations and one fp32 scale per token
              (SparseMatrix.linear_w8a8).
  stack       one decode step of a stack of Llama-2-7B layers (LinearStack), replayed as the CUDA
              graph that the program captured once.
  update      the masked weight step of sparse training on the compressed weight, and the updated
              dense weight read back (masked_update, decompress).
  decompress  the dense masked weight of a compressed layer (export, evaluation, re-pruning).
  compress    compressing a pruned layer when it is loaded, read back dense.

The sizes of the listed cases are the Llama-2-7B shapes that the benchmark and the tests use, and
one generic ragged shape; `draw` spreads sizes, sparsities (50 to 80 %), value types and batch
sizes over the range between and around them.
"""
import math

import numpy as np
import torch

from paper_2405_03594_gb300 import sp
from paper_2405_03594_gb300.stack import D_FF, D_MODEL, STACK_WEIGHT_STD, LinearStack

# Llama-2-7B linear shapes [N, K], as the benchmark names them
SHAPES = {"qkv": (12288, 4096), "o": (4096, 4096), "gate_up": (22016, 4096), "down": (4096, 11008)}
WEIGHT_STD = 0.02
LR = 1e-3


def listed():
    """The cases in order of their work."""
    return [
        # the smallest call of a decode step: one token through the attention output projection
        _layer("o_m1_bf16", "linear", "o", m=1, pct=70, dtype="bf16"),
        # one token through the widest layer, weights quantized to INT8
        _layer("gate_up_m1_int8", "linear", "gate_up", m=1, pct=70, dtype="int8"),
        # four sequences decoded together
        _layer("gate_up_m4_bf16", "linear", "gate_up", m=4, pct=70, dtype="bf16"),
        # sixteen sequences, the long-K layer, the lowest sparsity of the range
        _layer("down_m16_bf16_50", "linear", "down", m=16, pct=50, dtype="bf16"),
        # a decode batch of the INT8 deployment: INT8 weights and activations
        _layer("qkv_m32_w8a8", "w8a8", "qkv", m=32, pct=70, dtype="int8"),
        # a whole decode step of four layers for one sequence, replayed as a CUDA graph
        {"name": "stack4_m1_bf16", "op": "stack", "layers": 4, "m": 1, "pct": 70, "dtype": "bf16"},
        # loading a pruned layer: dense weight and mask to the compressed form (read back dense)
        _layer("o_compress_bf16", "compress", "o", m=0, pct=70, dtype="bf16"),
        # exporting the widest layer as a dense weight
        _layer("gate_up_decompress_bf16", "decompress", "gate_up", m=0, pct=70, dtype="bf16"),
        # one optimizer step of sparse training on the long-K layer, and its weight read back
        _layer("down_update_bf16", "update", "down", m=0, pct=70, dtype="bf16"),
        # a short ragged prompt through a layer whose sizes are multiples of no tile
        {"name": "ragged_m333_bf16", "op": "linear", "n": 5003, "k": 3656, "m": 333, "pct": 60, "dtype": "bf16"},
        # a chunk of a chunked prefill, INT8 weights
        _layer("qkv_m256_int8", "linear", "qkv", m=256, pct=60, dtype="int8"),
        # the prefill of a 2048-token prompt through the widest layer
        _layer("gate_up_m2048_bf16", "linear", "gate_up", m=2048, pct=70, dtype="bf16"),
    ]


def _layer(name, op, shape, m, pct, dtype):
    n, k = SHAPES[shape]
    return {"name": name, "op": op, "n": n, "k": k, "m": m, "pct": pct, "dtype": dtype}


def draw(rng):
    """One more case of the listed ranges: N 256 ... 22016, K 256 ... 11008 (a multiple of 8),
    M 1 ... 2048, sparsity 50 ... 80 %."""
    op = rng.choice(["linear"] * 8 + ["w8a8"] * 2 + ["stack", "update", "decompress", "compress"])
    pct = rng.randint(50, 80)
    if op == "stack":
        return {"op": "stack", "layers": rng.randint(1, 4), "m": _log_int(rng, 1, 64), "pct": pct,
                "dtype": rng.choice(["bf16", "int8"])}
    if rng.random() < 0.4:
        n, k = rng.choice(sorted(SHAPES.values()))
    else:
        n, k = _log_int(rng, 256, 22016), 8 * _log_int(rng, 32, 1376)
    k = max(256, min(k, 22016 * 4096 // n // 8 * 8))  # no larger than the largest listed layer
    m = 0 if op in ("update", "decompress", "compress") else _log_int(rng, 1, 2048)
    dtype = "int8" if op == "w8a8" else "bf16" if op == "update" else rng.choice(["bf16", "bf16", "int8"])
    return {"op": op, "n": n, "k": k, "m": m, "pct": pct, "dtype": dtype}


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1))


def _normal(shape, g, std=1.0):
    """std * N(0, 1) in bf16."""
    return torch.randn(shape, generator=g, device="cuda").mul_(std).to(torch.bfloat16)


def _keep_mask(w, pct):
    """uint8 keep-mask: in each row the pct % entries of smallest magnitude are dropped."""
    k = w.shape[1]
    drop = round(pct * k / 100)
    thr = torch.empty((w.shape[0], 1), dtype=w.dtype, device=w.device)
    for r in range(0, w.shape[0], 4096):
        thr[r:r + 4096] = w[r:r + 4096].abs().kthvalue(drop, dim=1, keepdim=True).values
    return (w.abs() > thr).to(torch.uint8)


def _weight(n, k, pct, dtype, g, std=WEIGHT_STD):
    """(values, mask, scale or None) of a pruned layer: bf16, or INT8 by absmax per row."""
    w = _normal((n, k), g, std)
    mask = _keep_mask(w, pct)
    if dtype == "bf16":
        return w, mask, None
    w = w.float() * mask
    amax = w.abs().amax(dim=1)
    s = torch.where(amax > 0, amax / 127.0, torch.ones_like(amax))
    q = torch.clamp(torch.round(w / s[:, None]), -127, 127).to(torch.int8)
    return q, mask, s


def _act_int8(x):
    """INT8 activations and one scale per token, by absmax."""
    xf = x.float()
    amax = xf.abs().amax(dim=1)
    sx = torch.where(amax > 0, amax / 127.0, torch.ones_like(amax))
    return torch.clamp(torch.round(xf / sx[:, None]), -127, 127).to(torch.int8), sx


def _inputs(case, seed):
    """Every tensor of a case but the stack's, from the seed alone."""
    g = _gen(seed)
    w, mask, s = _weight(case["n"], case["k"], case["pct"], case["dtype"], g)
    out = {"w": w, "mask": mask, "s": s}
    if case["op"] in ("linear", "w8a8"):
        out["x"] = _normal((case["m"], case["k"]), g)
        if case["op"] == "w8a8":
            out["qx"], out["sx"] = _act_int8(out["x"])
    if case["op"] == "update":
        out["grad"] = torch.randn((case["n"], case["k"]), generator=g, device="cuda")
    return out


def _stack_inputs(case, seed):
    """One layer's {name: (values, mask, scale)} on the GPU and the step's input rows."""
    g = _gen(seed)
    layer = {name: _weight(*SHAPES[name], case["pct"], case["dtype"], g, STACK_WEIGHT_STD) for name in SHAPES}
    return layer, _normal((case["m"], D_MODEL), g)


def _to_host(t):
    return None if t is None else (t.view(torch.int16) if t.dtype == torch.bfloat16 else t).cpu().numpy()


# ------------------------------------------------------------------ the program
def prepare(case, seed):
    if case["op"] == "stack":
        layer, x = _stack_inputs(case, seed)
        host = {name: tuple(_to_host(t) for t in v) for name, v in layer.items()}
        host = {name: (v.view("uint16") if v.dtype == "int16" else v, m, s) for name, (v, m, s) in host.items()}
        st = LinearStack(layers=case["layers"], pct=case["pct"], int8=case["dtype"] == "int8", max_m=case["m"],
                         host=host)
        st.set_input(x)
        return {"op": "stack", "stack": st, "graph": st.capture(case["m"]), "m": case["m"]}
    t = _inputs(case, seed)
    if case["op"] == "compress":
        return {"op": "compress", **t}
    h = sp.compress(t["w"], t["mask"], t["s"])
    state = {"op": case["op"], "h": h}
    if case["op"] == "linear":
        state["x"] = t["x"]
        state["ws"] = torch.zeros(max(h.workspace_size(case["m"]), 256), dtype=torch.uint8, device="cuda")
    elif case["op"] == "w8a8":
        state["qx"], state["sx"] = t["qx"], t["sx"]
        state["ws"] = torch.zeros(max(h.w8a8_workspace_size(case["m"]), 256), dtype=torch.uint8, device="cuda")
    elif case["op"] == "update":
        state["grad"] = t["grad"]
    return state


def run(state):
    op = state["op"]
    if op == "linear":
        return state["h"].linear(state["x"], workspace=state["ws"])
    if op == "w8a8":
        return state["h"].linear_w8a8(state["qx"], state["sx"], workspace=state["ws"])
    if op == "stack":
        state["graph"].replay()
        st, m = state["stack"], state["m"]
        # the hidden state, and the last layer's fused q/k/v
        return st.h[:m], st.qkv[:m]
    if op == "update":
        state["h"].masked_update(state["grad"], LR)
        return state["h"].decompress()
    if op == "decompress":
        return state["h"].decompress()
    return sp.compress(state["w"], state["mask"], state["s"]).decompress()


# ------------------------------------------------------------------ what is expected
def work(case):
    """Bytes: the compressed weight (kept values and one mask bit per entry), inputs and outputs
    once each; flops: one multiply-add per kept weight and row."""
    if case["op"] == "stack":
        one = [_linear_work(*SHAPES[name], case["pct"], case["dtype"], case["m"]) for name in SHAPES]
        return {"bytes": case["layers"] * sum(b for b, _ in one), "flops": case["layers"] * sum(f for _, f in one)}
    n, k, es = case["n"], case["k"], _esize(case)
    comp = _compressed_bytes(n, k, case["pct"], case["dtype"])
    kept = n * (k - round(case["pct"] * k / 100))
    if case["op"] == "linear":
        b, f = _linear_work(n, k, case["pct"], case["dtype"], case["m"])
        return {"bytes": b, "flops": f}
    if case["op"] == "w8a8":
        return {"bytes": comp + case["m"] * (k + 4 + 2 * n), "flops": 2 * case["m"] * kept}
    if case["op"] == "update":  # the gradient, the kept values read and written; the weight read back
        return {"bytes": 4 * n * k + comp + 2 * kept + 2 * n * k, "flops": 2 * kept}
    if case["op"] == "decompress":
        return {"bytes": comp + es * n * k, "flops": 0}
    # the dense weight and its mask in, the compressed form out and in again, the dense weight out
    return {"bytes": (es + 1) * n * k + 2 * comp + es * n * k, "flops": 0}


def _esize(case):
    return 2 if case["dtype"] == "bf16" else 1


def _compressed_bytes(n, k, pct, dtype):
    kept = n * (k - round(pct * k / 100))
    return kept * (2 if dtype == "bf16" else 1) + n * k // 8 + (0 if dtype == "bf16" else 4 * n)


def _linear_work(n, k, pct, dtype, m):
    kept = n * (k - round(pct * k / 100))
    return _compressed_bytes(n, k, pct, dtype) + 2 * m * (k + n), 2 * m * kept


def tolerance(case):
    """Exact where only stored values move or are rounded once elementwise; else about four times
    the distance from the 64-bit result: one bf16 rounding of the output (a linear), one more per
    activation (INT8 activations), or one per linear and residual add of the step (a stack)."""
    if case["op"] in ("update", "decompress", "compress"):
        return "exact"
    if case["op"] == "w8a8":
        return {"rel": 1e-2, "max": 4.5e-2}
    if case["op"] == "stack":
        return {"rel": 1.5e-2}
    return {"rel": 7e-3, "max": 1.6e-2}


def exact(case, seed):
    """The same results in 64 bits."""
    if case["op"] == "stack":
        return _exact_stack(case, seed)
    t = _inputs(case, seed)
    w = t["w"].double()
    if case["op"] == "update":
        w = w - LR * t["grad"].double()
    w *= t["mask"]
    if case["op"] in ("update", "decompress", "compress"):
        return w
    if t["s"] is not None:
        w *= t["s"].double()[:, None]
    x = t["qx"].double() * t["sx"].double()[:, None] if case["op"] == "w8a8" else t["x"].double()
    return x @ w.T


def _exact_stack(case, seed):
    layer, x = _stack_inputs(case, seed)
    w = {}
    for name, (v, mask, s) in layer.items():
        w[name] = v.double() * mask
        if s is not None:
            w[name] *= s.double()[:, None]
    # the stack's fixed residual vectors: N(0, 1) in bf16, two per layer, from its default seed
    rng = np.random.default_rng(np.random.SeedSequence([0, 0, 9, 3]))
    r = torch.from_numpy(rng.standard_normal((2 * case["layers"], D_MODEL), dtype=np.float32)).cuda()
    r = r.to(torch.bfloat16).double()
    h = x.double()
    qkv = None
    for l in range(case["layers"]):
        qkv = h @ w["qkv"].T
        h = h + qkv[:, 2 * D_MODEL:] @ w["o"].T + r[2 * l]
        gu = h @ w["gate_up"].T
        h = h + (gu[:, :D_FF] * gu[:, D_FF:]) @ w["down"].T + r[2 * l + 1]
    return h, qkv
