"""The calls that the speed of this library is judged by: what users have it do, from the smallest call to the largest.

`listed()` holds the fixed cases and `draw()` gives more of the same ranges; `prepare()` makes what a program has in hand
before the call, `run()` is one call of the public API, `work()` what that call cannot do without.  Four operations:

* ``weights``    ``attnw_fused``: attention weights from queries and keys, bfloat16 or float32
* ``rows``       ``softmax_rows``: row Softmax of float32 scores, bfloat16 or float32 result
* ``attention``  ``attn_fused``: the weights times the values
* ``project``    ``project_qk``: queries and keys of all heads from the layer's input
"""
from __future__ import annotations

import math

import torch

from paper_2407_13885_b200 import binding

_ELEMENTS = 1 << 31  # attention weights of the largest call
_DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _weights(name, B, H, N, d, out="bf16", sigma=1.0):
    return {"name": name, "op": "weights", "B": B, "H": H, "N": N, "d": d, "out": out, "sigma": sigma}


def _attention(name, B, H, N, d, sigma=1.0):
    return {"name": name, "op": "attention", "B": B, "H": H, "N": N, "d": d, "out": "bf16", "sigma": sigma}


def _rows(name, rows, cols, out="bf16"):
    return {"name": name, "op": "rows", "rows": rows, "cols": cols, "out": out, "sigma": 3.0}


def _project(name, B, N, d_model, H, d):
    return {"name": name, "op": "project", "B": B, "N": N, "d_model": d_model, "H": H, "d": d, "out": "bf16"}


def listed():
    return [
        # One head of a short sequence with float32 weights, the smallest configuration: the latency of a call.
        _weights("weights_f32_1x256", 1, 1, 256, 64, "f32"),
        # A 12-head layer on one sequence of 2048: an ordinary inference call.
        _weights("weights_bf16_12x2048", 1, 12, 2048, 64),
        # The headline: a 32-head layer on a batch of four sequences of 4096, 4.3 GB of weights.
        _weights("weights_bf16_128x4096", 4, 32, 4096, 128),
        # A long sequence with large logits (peaked rows), beyond what stays on chip.
        _weights("weights_bf16_8x16384", 1, 8, 16384, 128, sigma=4.0),
        # A small batch whose length no tile divides.
        _weights("weights_bf16_24x1000", 2, 12, 1000, 64),
        # float32 weights for analysis (attention maps, distillation targets), ragged length.
        _weights("weights_f32_16x2052", 1, 16, 2052, 128, "f32"),
        # Precomputed scores of eight heads over 8192 keys: the dedicated Softmax at the size it is quoted on.
        _rows("rows_bf16_32768x8192", 8 * 4096, 8192),
        # Short ragged rows, float32 in and out: classifier or router logits of one batch.
        _rows("rows_f32_4096x1000", 4096, 1000, "f32"),
        # Very long rows: logits over a large vocabulary or a long context.
        _rows("rows_bf16_2048x131072", 2048, 131072),
        # The whole attention layer at the headline's size.
        _attention("attention_128x4096", 4, 32, 4096, 128),
        # The whole attention layer of a small model on one ragged sequence.
        _attention("attention_12x1021", 1, 12, 1021, 64),
        # Queries and keys of all heads in front of the headline call.
        _project("project_4x4096_to_32x128", 4, 4096, 4096, 32, 128),
    ]


def _log_uniform(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def _heads(rng, N, most):
    """Batch and heads, spread over their logarithm up to what the largest call holds."""
    bh = _log_uniform(rng, 1, max(1, min(128, most // (N * N))))
    B = rng.choice([b for b in (1, 2, 3, 4) if bh % b == 0])
    return B, bh // B


def draw(rng):
    op = rng.choice(["weights", "weights", "weights", "rows", "rows", "attention", "attention", "project"])
    if op == "weights":
        out = rng.choice(["bf16", "bf16", "bf16", "f32"])
        step = 8 if out == "bf16" else 4
        N = max(64, _log_uniform(rng, 64, 16384) // step * step)
        B, H = _heads(rng, N, _ELEMENTS if out == "bf16" else _ELEMENTS // 2)
        case = _weights("", B, H, N, rng.choice([64, 128]), out, rng.choice([1.0, 1.0, 4.0]))
    elif op == "attention":
        N = _log_uniform(rng, 64, 16384)
        B, H = _heads(rng, N, _ELEMENTS)
        case = _attention("", B, H, N, rng.choice([64, 128]), rng.choice([1.0, 1.0, 4.0]))
    elif op == "rows":
        cols = max(64, _log_uniform(rng, 64, 262144) // 4 * 4)
        rows = _log_uniform(rng, max(1, (1 << 16) // cols), max(2, (1 << 28) // cols))
        case = _rows("", rows, cols, rng.choice(["bf16", "bf16", "f32"]))
    else:
        d = rng.choice([64, 128])
        H = _log_uniform(rng, 4, 4096 // d)
        d_model = rng.choice([H * d, H * d, 8 * _log_uniform(rng, 32, 512)])
        case = _project("", rng.choice([1, 1, 2, 4]), _log_uniform(rng, 64, 4096), d_model, H, d)
    del case["name"]
    return case


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def normal(*shape, sigma=1.0, dtype=torch.bfloat16):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=dtype).mul_(sigma)

    state = {"op": case["op"], "out": _DTYPES[case["out"]]}
    if case["op"] == "rows":
        state["S"] = normal(case["rows"], case["cols"], sigma=case["sigma"], dtype=torch.float32)
    elif case["op"] == "project":
        state["X"] = normal(case["B"], case["N"], case["d_model"])
        for w in ("Wq", "Wk"):  # unit-variance queries and keys
            state[w] = normal(case["H"], case["d"], case["d_model"], sigma=case["d_model"] ** -0.5)
    else:
        shape = (case["B"], case["H"], case["N"], case["d"])
        state["Q"], state["K"] = normal(*shape, sigma=case["sigma"]), normal(*shape, sigma=case["sigma"])
        state["scale"] = case["d"] ** -0.5
        if case["op"] == "attention":
            state["V"] = normal(*shape)
    return state


def run(state):
    op = state["op"]
    if op == "weights":
        return binding.attnw_fused(state["Q"], state["K"], state["scale"], out_dtype=state["out"])
    if op == "rows":
        return binding.softmax_rows(state["S"], out_dtype=state["out"])
    if op == "attention":
        return binding.attn_fused(state["Q"], state["K"], state["V"], state["scale"])
    return binding.project_qk(state["X"], state["Wq"], state["Wk"])


def work(case):
    out_bytes = 2 if case["out"] == "bf16" else 4
    if case["op"] == "rows":
        n = case["rows"] * case["cols"]
        return {"bytes": n * (4 + out_bytes), "flops": 0}
    if case["op"] == "project":
        x = case["B"] * case["N"] * case["d_model"]
        w = 2 * case["H"] * case["d"] * case["d_model"]
        qk = 2 * case["B"] * case["N"] * case["H"] * case["d"]
        return {"bytes": 2 * (x + w + qk), "flops": 2 * qk * case["d_model"]}
    bh, N, d = case["B"] * case["H"], case["N"], case["d"]
    if case["op"] == "weights":
        return {"bytes": bh * (2 * N * d * 2 + N * N * out_bytes), "flops": 2 * bh * N * N * d}
    return {"bytes": bh * 4 * N * d * 2, "flops": 4 * bh * N * N * d}


def tolerance(case):
    """About four times what the results differ by from the same formulas in 64 bits: over the listed cases and fifty more
    float32 results by 8e-7 and 1.9e-5 (large logits: the tensor cores' float32 sums), bfloat16 ones by 1.7e-3 and
    4.8e-3 (one rounding), attention by 2.4e-3 and 1.3e-2 (weights and result both rounded)."""
    if case["out"] == "f32":
        return {"rel": 4e-6, "max": 8e-5}
    if case["op"] == "attention":
        return {"rel": 1e-2, "max": 5e-2}
    return {"rel": 7e-3, "max": 2e-2}
