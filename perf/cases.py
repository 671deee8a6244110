"""The calls whose speed matters to a user of this library, as timed cases.

A case is one pass through the public entry points of ``paper_2404_07904_b200.binding``, as a training step, a
prefill or a decode loop makes it.  ``kind`` says which:

* ``train``   ``hgrn2_fwd`` and then ``hgrn2_bwd`` of one layer,
* ``packed``  the same through ``hgrn2_*_varlen`` on sequences of unequal length laid end to end,
* ``gated``   the same through ``hgrn2_*_gated`` (pre-activations in, their gradients out),
* ``prefill`` ``hgrn2_fwd`` for inference: nothing is kept for a backward, the final state is,
* ``step``    ``hgrn2_step``: one token for every sequence of a decode batch,
* ``burst``   ``hgrn2_step_multi``: several tokens for every sequence of a decode batch.

``io`` is the element type of the sequence tensors, ``B, H, N, d`` are batch, heads, tokens and head size
(d_k = d_v = d: the layer's expand ratio), ``gamma`` is the lower bound of the forget gates and ``state`` says whether an
initial state and a gradient of the final state come in.
"""
from __future__ import annotations

import math

import torch

from paper_2404_07904_b200 import binding

_DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def listed():
    def case(name, kind, B, H, N, d=128, io="bf16", gamma=0.9, state=False, **more):
        return dict(name=name, kind=kind, io=io, B=B, H=H, N=N, d=d, gamma=gamma, state=state, **more)

    return [
        # one user at the prompt: one token of one sequence, 16 heads - the smallest call, all latency
        case("decode_one", "step", 1, 16, 1),
        # a serving batch: one token for 256 sequences, the states (268 MB) cross the memory bus once each way
        case("decode_256", "step", 256, 16, 1),
        # the same batch checking eight drafted tokens per call
        case("decode_burst_8", "burst", 256, 16, 8),
        # a prompt of 5000 tokens (no whole number of chunks), one sequence: few long chains
        case("prefill_5000", "prefill", 1, 16, 5000, gamma=0.99),
        # training step of the 1B model's layer (hidden 2048, sequences of 2048): the headline
        case("train_lm_2048", "train", 8, 16, 2048),
        # the 2.9B model's layer (hidden 2560) at twice the context: 160 chains
        case("train_lm_2560", "train", 8, 20, 4096, gamma=0.5),
        # long-context training, 16 K tokens, states handed over between calls
        case("train_long_16k", "train", 2, 16, 16384, gamma=0.99, state=True),
        # long-context fine-tuning on a packed batch: 24 sequences of 4096 ... 256 tokens
        case("train_packed_mix", "packed", 24, 16, 4096, shortest=256),
        # the 1B model's layer from its projections' outputs (activations inside the call)
        case("train_gated_2048", "gated", 8, 16, 2048),
        # float32 at the size of a unit test or a toy model: short chains, few of them
        case("train_tiny_f32", "train", 1, 2, 256, d=64, io="f32", gamma=0.5),
        # the 1B model's layer in float32: a precision check, or a run that does not trust bf16
        case("train_f32_2048", "train", 2, 16, 2048, io="f32"),
        # a small model with heads of 64 in bf16 (hidden 1024)
        case("train_bf16_d64", "train", 4, 16, 2048, d=64),
    ]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    """One more case of the same ranges.  Token counts are spread over their logarithm and are whatever comes out
    (whole chunks are rare in serving, usual in training: about half of the training draws are rounded to them)."""
    kind = rng.choice(("train", "train", "train", "prefill", "step", "burst", "packed", "gated", "fp32", "small_d"))
    H = rng.choice((6, 8, 12, 16, 20))            # hidden sizes 768 ... 2560 at an expand ratio of 128
    gamma = rng.choice((0.0, 0.5, 0.9, 0.99))
    case = dict(kind=kind, io="bf16", B=1, H=H, N=1, d=128, gamma=gamma, state=rng.random() < 0.3)
    if kind in ("step", "burst"):
        case.update(B=_log_int(rng, 1, 256), N=1 if kind == "step" else rng.randint(2, 16), state=True,
                    io=rng.choice(("bf16", "bf16", "f32")), d=rng.choice((64, 128, 128)))
        return case
    if kind in ("fp32", "small_d"):
        # the float32 kernels: any head size in float32, the smaller ones in bf16
        case.update(kind="train", io="f32" if kind == "fp32" else "bf16",
                    d=rng.choice((64, 128)) if kind == "fp32" else rng.choice((32, 64)), N=_log_int(rng, 64, 2048))
        most = 2 * 16 * 2048
    else:
        case["N"] = _log_int(rng, 48, 16384)
        most = 8 * 20 * 4096
    if kind == "packed":
        case["B"] = rng.randint(2, 32)
        case["N"] = max(64, min(case["N"], 8192, most // (H * case["B"])))
        case["shortest"] = rng.randint(1, case["N"])
        return case
    if kind != "prefill" and rng.random() < 0.5:
        case["N"] = max(64, case["N"] // 64 * 64)
    case["B"] = _log_int(rng, 1, max(1, min(32, most // (H * case["N"]))))
    return case


def _lengths(case):
    """Sequence lengths of a packed batch, longest first, in equal ratios from N down to `shortest`."""
    n, lo, hi = case["B"], case["shortest"], case["N"]
    return [int(round(hi * (lo / hi) ** (j / max(1, n - 1)))) for j in range(n)]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    io, B, H, N, d = _DTYPES[case["io"]], case["B"], case["H"], case["N"], case["d"]
    kind, gamma, scale = case["kind"], case["gamma"], d ** -0.5

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)

    if kind == "packed":
        lens = _lengths(case)
        seq = (H, sum(lens), d)
    elif kind == "step":
        seq = (B, H, d)
    else:
        seq = (B, H, N, d)
    s = {"kind": kind, "S0": None, "dSN": None}
    if kind == "gated":
        for name in ("zo", "zf", "zi"):
            s[name] = normal(*seq).to(io)
        s["beta"] = gamma + (0.95 - gamma) * torch.rand((H, d), generator=gen, device="cuda") if gamma < 0.95 else \
            torch.full((H, d), gamma, device="cuda")
    else:
        s["o"] = (normal(*seq) * scale).to(io)
        s["f"] = (gamma + (1 - gamma) * torch.sigmoid(normal(*seq))).to(io)
        s["i"] = (normal(*seq) * scale).to(io)
    if kind in ("train", "packed", "gated"):
        s["dy"] = normal(*seq).to(io)
    if kind in ("step", "burst"):
        s["S"] = normal(B, H, d, d) * 0.02
        s["y"] = torch.empty(seq, dtype=io, device="cuda")
    elif case["state"]:
        s["S0"] = normal(B, H, d, d) * 0.02
        if kind != "prefill":
            s["dSN"] = normal(B, H, d, d) * 0.02
    if kind == "packed":
        starts = [0]
        for n in lens:
            starts.append(starts[-1] + n)
        s["cu"] = torch.tensor(starts, dtype=torch.int32, device="cuda")
    return s


def run(s):
    kind = s["kind"]
    if kind == "step":
        return binding.hgrn2_step(s["o"], s["f"], s["i"], s["S"], y=s["y"]), s["S"]
    if kind == "burst":
        return binding.hgrn2_step_multi(s["o"], s["f"], s["i"], s["S"], y=s["y"]), s["S"]
    if kind == "prefill":
        y, SN, _, _, _ = binding.hgrn2_fwd(s["o"], s["f"], s["i"], s["S0"], save_for_backward=False)
        return y, SN
    if kind == "train":
        y, SN, saved, ws, _ = binding.hgrn2_fwd(s["o"], s["f"], s["i"], s["S0"])
        d_o, d_f, d_i, dS0, _ = binding.hgrn2_bwd(s["o"], s["f"], s["i"], s["S0"], s["dy"], s["dSN"], saved, ws=ws)
        return y, SN, d_o, d_f, d_i, dS0
    if kind == "packed":
        y, SN, saved, ws, _ = binding.hgrn2_fwd_varlen(s["o"], s["f"], s["i"], s["cu"], s["S0"])
        d_o, d_f, d_i, dS0, _ = binding.hgrn2_bwd_varlen(s["o"], s["f"], s["i"], s["cu"], s["S0"], s["dy"], s["dSN"],
                                                         saved, ws=ws)
        return y, SN, d_o, d_f, d_i, dS0
    y, SN, saved, ws, _ = binding.hgrn2_fwd_gated(s["zo"], s["zf"], s["zi"], s["beta"], s["S0"])
    d_zo, d_zf, d_zi, d_beta, dS0, _ = binding.hgrn2_bwd_gated(s["zo"], s["zf"], s["zi"], s["beta"], s["S0"], s["dy"],
                                                               s["dSN"], saved, ws=ws)
    return y, SN, d_zo, d_zf, d_zi, d_beta, dS0


def work(case):
    """Each input read once and each output written once; operations of the recurrence itself for the decode calls
    (decay, outer product and output: 5 per state element and token) and of its chunkwise form (causal count, chunks
    of 64) for the others."""
    kind, B, H, N, d = case["kind"], case["B"], case["H"], case["N"], case["d"]
    size = 2 if case["io"] == "bf16" else 4
    rows = H * sum(_lengths(case)) if kind == "packed" else B * H * N
    state = B * H * d * d * 4
    if kind in ("step", "burst"):
        return {"bytes": 2 * state + 4 * rows * d * size, "flops": 5 * rows * d * d}
    fwd = rows * (4 * d * d + 2 * d * 65)
    ins = state if case["state"] else 0
    if kind == "prefill":
        return {"bytes": 4 * rows * d * size + state + ins, "flops": fwd}
    return {"bytes": 11 * rows * d * size + 2 * state + 3 * ins + (8 * H * d if kind == "gated" else 0),
            "flops": fwd + rows * (8 * d * d + 5 * d * 65)}


def tolerance(case):
    if case["io"] == "f32":
        return {"rel": 1e-5, "max": 2e-4}         # sums of float32 products, in whatever order; d_f divides by f
    if case["kind"] in ("step", "burst") or case["d"] != 128:
        return {"rel": 2e-3, "max": 1.6e-2}       # computed in float32, rounded to bf16 where written
    return {"rel": 1e-2, "max": 0.1}              # bf16 operands, float32 sums and state
