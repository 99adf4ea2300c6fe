"""Performance cases of the P-EAGLE drafter-attention library: the calls that a training program
makes, through the public entry points of ``paper_2602_01469_b200.binding``.

A case names one of six ways in which the library is used (``"call"``):

  step        ``peagle_attn_partitioned``: forward and backward of a batch, the hot path of training
  forward     ``peagle_attn_fwd`` (or ``peagle_attn_fwd_static``) per partition: validation loss
  autograd    ``peagle_attn_fwd`` per partition, later ``peagle_attn_bwd`` per partition into fp32
              sums and ``peagle_cast_grads``: how an autograd function of a framework calls it
  layer       ``peagle_layer_partitioned``: projection, rotary and attention, segment by segment
  projection  ``peagle_gemm_bf16`` and ``peagle_rope_qkv_fwd / _bwd``: the same prologue and its
              backward for a program that strings the pieces together itself
  host        ``peagle_attn_partitioned_host``: the step with its tensors in pinned host memory

Head counts and head sizes are those of the benchmark's workloads and of the tests; lengths run from
a few dozen context tokens to the 90th percentile of the reasoning traces (11,008) and to batches
of a long-tail mixture; depths, segment counts, memory orders and COD retention as in ``inputs``.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2602_01469_b200 import binding, inputs

ROPE_BASE = 500000.0
D_MODEL = 2880

GPTOSS = {"q_heads": 64, "kv_heads": 8, "head_dim": 64}
QWEN3CODER = {"q_heads": 32, "kv_heads": 4, "head_dim": 128}
TINY = {"q_heads": 4, "kv_heads": 1, "head_dim": 64}
# further shapes that the tests run: an odd group of query heads per KV head, one query head per
# KV head, more KV heads than the one-key-per-row path takes
ODD_GROUP = {"q_heads": 3, "kv_heads": 1, "head_dim": 64}
NO_GROUP = {"q_heads": 24, "kv_heads": 24, "head_dim": 64}
SMALL_128 = {"q_heads": 8, "kv_heads": 2, "head_dim": 128}


def _case(call, n, heads, *, name=None, K=8, segments=1, seg_len=0, cod_r=0.0, order="depth_major",
          batch_tokens=0, length_seed=0, d_model=0, entry="context"):
    """A case as plain values.  ``n``: context tokens of the one sequence; 0 with ``batch_tokens``:
    a batch of sequences with long-tail lengths, that many context tokens in all."""
    c = {"call": call, "n": n, "K": K, **heads, "segments": segments, "seg_len": seg_len, "cod_r": cod_r,
         "order": order, "batch_tokens": batch_tokens, "length_seed": length_seed, "d_model": d_model,
         "entry": entry}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # a unit-test sized step: the time is launches and host work, as for any very short example
        _case("step", 128, TINY, name="step_tiny", K=4),
        # a short prompt of odd length at the Qwen3-Coder-like layer shape: most tiles are ragged
        _case("step", 391, QWEN3CODER, name="step_short_d128"),
        # the Qwen3-Coder-like layer at half the median trace length, the usual step at head size 128
        _case("step", 2048, QWEN3CODER, name="step_qwen_n2048"),
        # the GPT-OSS-like layer at the median trace length: the benchmark's headline step
        _case("step", 4096, GPTOSS, name="step_gptoss_n4096"),
        # the paper's own example of COD down-sampling: 8,192 tokens, retention 0.8, ragged depth blocks
        _case("step", 8192, GPTOSS, name="step_gptoss_cod_n8192", cod_r=0.8),
        # a 90th-percentile trace in four segments, the largest single example
        _case("step", 11008, GPTOSS, name="step_p90_s4", segments=4),
        # a batch of long-tail lengths (ragged, some of them short) in 8,192-token segments
        _case("step", 0, GPTOSS, name="step_longtail_batch", seg_len=8192, batch_tokens=65536),
        # validation: only the forward of a median-length trace (the median itself, an odd length)
        _case("forward", 3891, GPTOSS, name="forward_n3891"),
        # forward and backward as separate calls of an autograd function, ordinary length, two segments
        _case("autograd", 1000, GPTOSS, name="autograd_n1000_s2", segments=2),
        # the attention half of the drafter layer at half the median length, two segments
        _case("layer", 2048, GPTOSS, name="layer_n2048_s2", segments=2, d_model=D_MODEL),
        # fused projection, rotary prologue and their backward over the headline's rows
        _case("projection", 4096, GPTOSS, name="projection_n4096", d_model=D_MODEL),
        # the step with its tensors in pinned host memory (activations offloaded to the host)
        _case("host", 2048, GPTOSS, name="host_gptoss_n2048"),
    ]


def _spread(rng, lo, hi):
    """A whole number from [lo, hi], even over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        call = rng.choices(("step", "forward", "autograd", "layer", "projection", "host"), (8, 2, 2, 2, 2, 1))[0]
        heads = rng.choices((GPTOSS, QWEN3CODER, TINY, ODD_GROUP, NO_GROUP, SMALL_128), (6, 5, 2, 1, 1, 2))[0]
        longest = {"step": 11008, "forward": 11008, "autograd": 8192, "layer": 4096, "projection": 4096, "host": 2048}
        n = _spread(rng, 24, longest[call])
        K = rng.choice((1, 2, 4, 6, 8, 8, 8))
        if call == "projection":
            c = _case(call, n, heads, K=K, d_model=8 * _spread(rng, 16, 512))
        elif call == "layer":
            c = _case(call, n, heads, K=K, segments=rng.randint(1, 3), d_model=8 * _spread(rng, 16, 512))
        elif call == "step" and rng.random() < 0.2:
            total = _spread(rng, 4096, 65536)
            c = _case(call, 0, heads, K=K, seg_len=rng.choice((2048, 4096, 8192)), batch_tokens=total,
                      length_seed=rng.randrange(1000))
        else:
            segments = rng.choice((1, 1, 2, 3, 4)) if n >= 64 else 1
            order = rng.choices(("depth_major", "anchor_major"), (5, 1))[0]
            cod_r = rng.choices((0.0, round(rng.uniform(0.6, 0.9), 2)), (4, 1))[0]
            c = _case(call, n, heads, K=K, segments=segments, order=order, cod_r=cod_r)
            if call == "forward" and segments == 1 and n * K <= 16384 and rng.random() < 0.4:
                c["entry"] = "static"
        if _cost(c) <= most:
            return c


def _cost(case):
    w = work(case)
    return max(w["bytes"] / 6.0e12, w["flops"] / 1.5e15)


# ------------------------------------------------------------------ sizes
def _lengths(case):
    if case["batch_tokens"]:
        return inputs.longtail_lengths(case["batch_tokens"], case["length_seed"])
    return (case["n"],)


def _workload(case, seed):
    return inputs.Workload("case", _lengths(case), case["K"], case["q_heads"], case["kv_heads"],
                           case["head_dim"], n_segments=case["segments"], seg_len=case["seg_len"] or None,
                           seed=seed, cod_r=case["cod_r"] or None, order=case["order"])


def _counts(case):
    """Expanded tokens and allowed (query, key) pairs: a token (anchor a, depth d) sees the a + 1 real
    tokens up to its anchor and its d chain tokens.  COD sets are drawn per seed; their sizes are fixed
    and their pairs move by a per cent or so, so those of one draw stand for all."""
    tokens = pairs = 0
    for i, n in enumerate(_lengths(case)):
        K = case["K"]
        if case["cod_r"]:
            a, d = inputs.cod_grid(n, K, case["cod_r"], i)
            tokens += a.shape[0]
            pairs += int(a.astype(np.int64).sum() + d.astype(np.int64).sum()) + a.shape[0]
        else:
            tokens += n * K
            pairs += K * n * (n + 1) // 2 + n * K * (K - 1) // 2
    return tokens, pairs


def work(case):
    """Bytes: every input read once, every output written once.  Flops: per allowed pair and query
    head 4 D forward and 10 D backward; the projection's three products."""
    T, P = _counts(case)
    Hq, Hkv, D, dm = case["q_heads"], case["kv_heads"], case["head_dim"], case["d_model"]
    q, kv = 2 * T * Hq * D, 2 * T * Hkv * D          # bytes of a query-side / key-side tensor
    lse, meta = 4 * T * Hq, 8 * T
    fwd, bwd = 4 * P * D * Hq, 10 * P * D * Hq
    width = (Hq + 2 * Hkv) * D
    call = case["call"]
    if call == "forward":
        return {"bytes": 2 * q + 2 * kv + lse + meta, "flops": fwd}
    if call in ("step", "autograd", "host"):
        return {"bytes": 4 * q + 4 * kv + lse + meta, "flops": fwd + bwd}
    if call == "layer":
        # X and dO in, O and dX out, W in and dW out; every segment projects the keys of the earlier
        # segments' depth-0 tokens again, which another schedule need not: not counted
        return {"bytes": 2 * (2 * T * dm) + 2 * q + 2 * (2 * width * dm) + lse + meta,
                "flops": fwd + bwd + 6 * T * width * dm}
    # projection: X, W and the gradients of Q, K, V in; Q, K, V, the fused rows' gradient and the fp32
    # gradients of X and W out
    return {"bytes": 2 * T * dm + 2 * width * dm + 3 * (q + 2 * kv) + 4 * T * dm + 4 * width * dm + meta,
            "flops": 6 * T * width * dm}


def tolerance(case):
    """bf16 inputs and outputs with fp32 accumulation; probabilities and their gradients pass through
    bf16 on the way to the tensor cores, as the parity tests allow for the gradients."""
    return {"rel": 1e-2}


# ------------------------------------------------------------------ what the program holds
@functools.lru_cache(maxsize=None)
def _context():
    """A training program keeps one context for its whole run."""
    return binding.Context(torch.cuda.current_device())


def _normal(gen, shape, std=1.0):
    return (torch.randn(shape, generator=gen, dtype=torch.bfloat16, device="cuda") * std)


def prepare(case, seed):
    call = case["call"]
    w = _workload(case, seed)
    cu, anchor, depth, parts = inputs.build_case(w, binding.peagle_assign_segments)
    T, Hq, Hkv, D, dm = int(cu[-1]), w.n_q_heads, w.n_kv_heads, w.head_dim, case["d_model"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    width = (Hq + 2 * Hkv) * D
    s = {"case": case, "ctx": _context(), "T": T, "width": width, "w": w,
         "parts": [binding.Partition(p["seq"], p["q"], p["k"]) for p in parts]}
    bf16 = {"dtype": torch.bfloat16, "device": "cuda"}
    f32 = {"dtype": torch.float32, "device": "cuda"}
    s["anchor"], s["depth"] = torch.from_numpy(anchor).cuda(), torch.from_numpy(depth).cuda()
    if call in ("layer", "projection"):
        s["X"] = _normal(gen, (T, dm))
        s["W"] = _normal(gen, (width, dm), 1.0 / math.sqrt(dm))
    if call == "projection":
        s["gQ"], s["gK"], s["gV"] = _normal(gen, (T, Hq, D)), _normal(gen, (T, Hkv, D)), _normal(gen, (T, Hkv, D))
        s["Y"], s["dY"] = torch.empty(T, width, **bf16), torch.empty(T, width, **bf16)
        s["Q"], s["K"], s["V"] = torch.empty(T, Hq, D, **bf16), torch.empty(T, Hkv, D, **bf16), torch.empty(T, Hkv, D, **bf16)
        s["dX"], s["dW"] = torch.empty(T, dm, **f32), torch.empty(width, dm, **f32)
        return s
    s["LSE"] = torch.empty(Hq, T, **f32)
    s["O"] = torch.empty(T, Hq, D, **bf16)
    if call == "layer":
        s["dO"] = _normal(gen, (T, Hq, D))
        s["dX"], s["dW"] = torch.empty(T, dm, **bf16), torch.empty(width, dm, **bf16)
    else:
        std = 1.0 / math.sqrt(D)
        s["Q"], s["K"], s["V"] = _normal(gen, (T, Hq, D), std), _normal(gen, (T, Hkv, D), std), _normal(gen, (T, Hkv, D), std)
        if call != "forward":
            s["dO"] = _normal(gen, (T, Hq, D))
            s["dQ"] = torch.empty(T, Hq, D, **bf16)
            s["dK"], s["dV"] = torch.empty(T, Hkv, D, **bf16), torch.empty(T, Hkv, D, **bf16)
        if call == "autograd":
            s["dK_acc"], s["dV_acc"] = torch.empty(T, Hkv, D, **f32), torch.empty(T, Hkv, D, **f32)
    if call == "host":
        for k in ("Q", "K", "V", "dO", "O", "LSE", "dQ", "dK", "dV"):
            h = torch.empty(s[k].shape, dtype=s[k].dtype, pin_memory=True)
            if k in ("Q", "K", "V", "dO"):
                h.copy_(s[k])
            s[k] = h
        s["prob"] = binding.Problem(cu, anchor, depth, w.K, Hq, Hkv, D, w.scale)
    else:
        s["prob"] = binding.Problem(cu, s["anchor"], s["depth"], w.K, Hq, Hkv, D, w.scale)
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    return _RUN[s["case"]["call"]](s)


def _step(s):
    binding.peagle_attn_partitioned(s["ctx"], s["prob"], s["parts"], s["Q"], s["K"], s["V"], s["dO"], s["O"],
                                    s["LSE"], s["dQ"], s["dK"], s["dV"])
    return [s["O"], s["LSE"], s["dQ"], s["dK"], s["dV"]]


def _host(s):
    binding.peagle_attn_partitioned_host(s["ctx"], s["prob"], s["parts"], s["Q"], s["K"], s["V"], s["dO"],
                                         s["O"], s["LSE"], s["dQ"], s["dK"], s["dV"])
    return [s["O"], s["LSE"], s["dQ"], s["dK"], s["dV"]]


def _forward(s):
    for p in s["parts"]:
        if s["case"]["entry"] == "static":
            binding.peagle_attn_fwd_static(0, s["prob"], p, s["Q"], s["K"], s["V"], s["O"], s["LSE"])
        else:
            binding.peagle_attn_fwd(s["ctx"], s["prob"], p, s["Q"], s["K"], s["V"], s["O"], s["LSE"])
    return [s["O"], s["LSE"]]


def _autograd(s):
    for p in s["parts"]:
        binding.peagle_attn_fwd(s["ctx"], s["prob"], p, s["Q"], s["K"], s["V"], s["O"], s["LSE"])
    s["dK_acc"].zero_()
    s["dV_acc"].zero_()
    for p in s["parts"]:
        binding.peagle_attn_bwd(s["ctx"], s["prob"], p, s["Q"], s["K"], s["V"], s["O"], s["dO"], s["LSE"],
                                s["dQ"], s["dK_acc"], s["dV_acc"])
    binding.peagle_cast_grads(s["ctx"], s["dK_acc"], s["dV_acc"], s["dK"], s["dV"])
    return [s["O"], s["LSE"], s["dQ"], s["dK"], s["dV"]]


def _layer(s):
    binding.peagle_layer_partitioned(s["ctx"], s["prob"], s["parts"], s["X"], s["W"], ROPE_BASE, s["dO"], s["O"],
                                     s["LSE"], s["dX"], s["dW"])
    return [s["O"], s["LSE"], s["dX"], s["dW"]]


def _projection(s):
    ctx, T, width, w, dm = s["ctx"], s["T"], s["width"], s["w"], s["case"]["d_model"]
    Hq, Hkv, D = w.n_q_heads, w.n_kv_heads, w.head_dim
    # Y = X W^T, split and rotated
    binding.peagle_gemm_bf16(ctx, s["X"], dm, 0, s["W"], dm, 0, s["Y"], width, 0, T, width, dm)
    binding.peagle_rope_qkv_fwd(ctx, s["Y"], s["anchor"], s["depth"], Hq, Hkv, D, ROPE_BASE, s["Q"], s["K"], s["V"])
    # gradients back through the rotation, then dX = dY W and dW = dY^T X into fp32 sums
    binding.peagle_rope_qkv_bwd(ctx, s["gQ"], s["gK"], s["gV"], s["anchor"], s["depth"], Hq, Hkv, D, ROPE_BASE, s["dY"])
    s["dX"].zero_()
    s["dW"].zero_()
    binding.peagle_gemm_bf16(ctx, s["dY"], width, 0, s["W"], dm, 1, s["dX"], dm, 1, T, dm, width)
    binding.peagle_gemm_bf16(ctx, s["dY"], width, 1, s["X"], dm, 1, s["dW"], dm, 1, width, dm, T)
    return [s["Q"], s["K"], s["V"], s["dY"], s["dX"], s["dW"]]


_RUN = {"step": _step, "forward": _forward, "autograd": _autograd, "layer": _layer, "projection": _projection,
        "host": _host}
