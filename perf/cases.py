"""The work that programs have this library do, as cases that can be timed: one pass each through the binding.

A layer case is one routed-expert feed-forward layer (route -> permute -> grouped SwiGLU GEMMs -> combine), forward only
(`pass` = "fwd"), a whole training step with the router's backward ("train"), or the expert-chunked training step that bounds the
activation memory ("chunked").  A vocabulary case is the projection with the online log-likelihood, forward ("vocab_fwd") or with
its gradients ("vocab_train").  Sizes are those of the library's own workloads (`synth.WORKLOADS`) and of its tests, or lie
between them; values have the distributions of `synth.make_inputs`.
"""
from __future__ import annotations

import math

import torch

from paper_2607_01844_b200 import binding, synth

SOFTMAX, SIGMOID = synth.SCORE_SOFTMAX, synth.SCORE_SIGMOID
NO_BIAS, POST_SCORE, PRE_LOGIT = synth.BIAS_NONE, synth.BIAS_POST_SCORE, synth.BIAS_PRE_LOGIT

# The widest forward layer: T k d f = 16384 * 8 * 7168 * 2048 multiply-adds per projection.  Drawn cases stay below its cost.
MOST_FLOPS = 6.0 * 16384 * 8 * 7168 * 2048
MOST_WEIGHT_BYTES = 23e9          # forward: bf16 weights; training: weights and fp32 gradients together
MOST_ROW_BYTES = 6e9              # expert-contiguous buffers and workspace


def _layer(name, T, d, E, k, f, what="fwd", score=SOFTMAX, bias=NO_BIAS, skew=False, recompute=False, chunks=0):
    c = {"pass": what, "T": T, "d": d, "E": E, "k": k, "f": f, "score": score, "bias": bias, "skew": skew,
         "recompute": recompute, "chunks": chunks}
    return {"name": name, **c} if name else c


def _vocab(name, what, N, H, V):
    c = {"pass": what, "N": N, "H": H, "V": V}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest layer of the test suite and the benchmark: launches and host calls are all there is
        _layer("fwd_tiny", 256, 256, 8, 2, 512),
        # decoding: a batch of 16 sequences, one token each, through a mid-size layer
        _layer("decode_mid", 16, 2048, 64, 6, 1408),
        # decoding through a trillion-scale layer: 64 tokens touch most of the 256 experts with two or three rows each
        _layer("decode_large", 64, 7168, 256, 8, 2048, score=SIGMOID, bias=POST_SCORE),
        # prefill or evaluation of a mid-size layer
        _layer("fwd_mid", 4096, 2048, 64, 6, 1408),
        # prefill of a trillion-scale layer with near-uniform load
        _layer("fwd_large", 16384, 7168, 256, 8, 2048, score=SIGMOID, bias=POST_SCORE),
        # the same layer under Zipf(1.2) load with a tenth of the experts empty (a router that has collapsed onto few experts)
        _layer("fwd_skew", 16384, 7168, 256, 8, 2048, score=SIGMOID, bias=POST_SCORE, skew=True),
        # training step of a mid-size layer, softmax router and its backward
        _layer("train_mid", 4096, 2048, 64, 6, 1408, "train"),
        # training step of a trillion-scale layer's share of experts: about 171 rows per expert, gradients dominate the traffic
        _layer("train_large", 2048, 7168, 96, 8, 2048, "train", score=SIGMOID, bias=POST_SCORE),
        # training step at widths that are multiples of 8 only, a token count that fits no tile, and a bias before the score
        _layer("train_odd", 1537, 1000, 20, 3, 1416, "train", score=SIGMOID, bias=PRE_LOGIT),
        # training step with expert-contiguous buffers for one quarter of the experts at a time (recomputes the up-projection)
        _layer("train_chunked", 4096, 7168, 64, 4, 2048, "chunked", score=SIGMOID, bias=POST_SCORE, chunks=4),
        # evaluation loss over a small vocabulary
        _vocab("vocab_eval", "vocab_fwd", 2048, 2048, 32000),
        # training step of the vocabulary projection at full hidden size and vocabulary
        _vocab("vocab_train", "vocab_train", 8192, 7168, 131072),
    ]


def _log(rng, lo, hi, step):
    """Log-uniform in [lo, hi], a multiple of `step`."""
    return max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))) / step) * step)


def draw(rng):
    """One more case of the same ranges: token counts from 1 on, any number of experts, widths in multiples of 64 and of 8."""
    while True:
        what = rng.choice(["decode", "decode", "fwd", "fwd", "fwd", "train", "train", "train", "chunked", "vocab_fwd", "vocab_train"])
        if what.startswith("vocab"):
            N, H, V = _log(rng, 256, 8192, 1), _log(rng, 512, 7168, 64), _log(rng, 8192, 131072, 64)
            if (2.0 if what == "vocab_fwd" else 8.0) * N * H * V <= MOST_FLOPS:
                return _vocab(None, what, N, H, V)
            continue
        step = 64 if what == "chunked" or rng.random() < 0.75 else 8
        d, f, E = _log(rng, 256, 7168, step), _log(rng, 256, 2048, step), _log(rng, 8, 256, 1)
        k = rng.randint(1, min(8, E))
        T = _log(rng, 1, 256, 1) if what == "decode" else _log(rng, 256, 16384, 1)
        score, bias = rng.choice([(SOFTMAX, NO_BIAS), (SIGMOID, NO_BIAS), (SIGMOID, POST_SCORE), (SIGMOID, PRE_LOGIT)])
        backward = what in ("train", "chunked")
        weights = 6.0 * E * d * f * (3 if backward else 1)
        rows = 2.0 * T * k * (2 * d + f) * (3 if backward else 1)
        flops = (22.0 if backward else 6.0) * T * k * d * f * (20 if step == 8 else 1)   # odd widths: on the CUDA cores' scale
        if weights > MOST_WEIGHT_BYTES or rows > MOST_ROW_BYTES or flops > MOST_FLOPS:
            continue
        return _layer(None, T, d, E, k, f, "fwd" if what == "decode" else what, score, bias,
                      recompute=what == "train" and rng.random() < 0.25, chunks=rng.randint(2, 8) if what == "chunked" else 0)


def _normal(shape, std, seed, dtype=torch.bfloat16):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    out = torch.empty(shape, dtype=dtype, device="cuda")
    flat = out.view(shape[0], -1)
    step = max(1, (1 << 27) // flat.shape[1])
    for r in range(0, shape[0], step):
        part = flat[r:r + step]
        part.copy_(torch.randn(part.shape, generator=g, device="cuda") * std)
    return out


def prepare(case, seed):
    if case["pass"].startswith("vocab"):
        N, H, V = case["N"], case["H"], case["V"]
        g = torch.Generator(device="cuda")
        g.manual_seed(seed * 31 + 5)
        st = {"case": case,
              "X": _normal((N, H), 1.0, seed * 31 + 1),
              "W": _normal((H, V), 0.02, seed * 31 + 2),
              "targets": torch.randint(0, V, (N,), generator=g, device="cuda", dtype=torch.int32),
              "loss": torch.empty(N, dtype=torch.float32, device="cuda"),
              "lse": torch.empty(N, dtype=torch.float32, device="cuda"),
              "ws": torch.empty(max(256, binding.mop_vocab_workspace_bytes(N, H, V)), dtype=torch.uint8, device="cuda")}
        if case["pass"] == "vocab_train":
            # upstream weight of a mean over the batch, some rows masked out
            st["dloss"] = -(torch.rand(N, generator=g, device="cuda") < 0.9).float() / N
            st["dX"] = torch.empty((N, H), dtype=torch.bfloat16, device="cuda")
            st["dW"] = torch.empty((H, V), dtype=torch.float32, device="cuda")
            st["ws_bwd"] = torch.empty(max(256, binding.mop_vocab_bwd_workspace_bytes(N, H, V)), dtype=torch.uint8, device="cuda")
        return st
    backward = case["pass"] != "fwd"
    w = synth.Workload("case", case["T"], case["d"], case["E"], case["k"], case["f"], case["score"], case["bias"],
                       0.01 if case["bias"] != NO_BIAS else 0.0, skew=case["skew"], backward=backward, seed=seed)
    st = {"case": case, "inp": synth.make_inputs(w, "cuda")}
    mode = 0 if not backward else 2 if case["recompute"] else 1
    st["ctx"] = binding.context_for(w, device=torch.cuda.current_device(), backward=mode)
    if case["pass"] == "chunked":
        T, d, E, k, f = w.T, w.d, w.E, w.k, w.f
        i32, b16, f32 = (dict(dtype=t, device="cuda") for t in (torch.int32, torch.bfloat16, torch.float32))
        st.update(idx=torch.empty((T, k), **i32), gate=torch.empty((T, k), **f32), counts=torch.empty((E,), **i32),
                  offsets=torch.empty((E + 1,), **i32), perm_row=torch.empty((T * k,), **i32),
                  row_src=torch.empty((T * k,), **i32), Y=torch.empty((T, d), **b16), dX=torch.empty((T, d), **b16),
                  dgate=torch.empty((T, k), **f32), dW_gate=torch.empty((E, d, f), **f32),
                  dW_up=torch.empty((E, d, f), **f32), dW_down=torch.empty((E, f, d), **f32))
        n = binding.mop_moe_chunked_workspace_bytes(st["ctx"], case["chunks"], True)
        st["ws"] = torch.empty(n, dtype=torch.uint8, device="cuda")
        return st
    st["buf"] = binding.LayerBuffers(w)
    if backward:
        st["logits"] = torch.empty((w.T, w.E), dtype=torch.float32, device="cuda")
        st["dW_r"] = torch.empty((w.d, w.E), dtype=torch.float32, device="cuda")
        st["dbias"] = torch.empty((w.E,), dtype=torch.float32, device="cuda") if w.bias_mode != NO_BIAS else None
        if case["recompute"]:
            st["buf"].G = st["buf"].U = None
    return st


def _train_step(st):
    ctx, inp, b = st["ctx"], st["inp"], st["buf"]
    binding.mop_moe_route(ctx, inp["x"], inp["W_r"], inp["bias"], b.idx, b.gate, st["logits"])
    binding.mop_moe_permute(ctx, inp["x"], b.idx, b.counts, b.offsets, b.perm_row, b.row_src, b.Xp)
    binding.mop_moe_expert_ffn_fwd(ctx, b.Xp, b.offsets, b.row_src, b.gate, inp["W_gate"], inp["W_up"], inp["W_down"],
                                   b.G, b.U, b.H, b.Yp)
    binding.mop_moe_combine(ctx, b.Yp, b.perm_row, b.Y)
    binding.mop_moe_expert_ffn_bwd(ctx, inp["dY"], b.Xp, b.G, b.U, None if st["case"]["recompute"] else b.H, b.offsets,
                                   b.perm_row, b.row_src, b.gate, inp["W_gate"], inp["W_up"], inp["W_down"], b.dX,
                                   b.dW_gate, b.dW_up, b.dW_down, b.dgate)
    binding.mop_moe_route_bwd(ctx, st["logits"], inp["bias"], b.idx, b.gate, b.dgate, b.Xp, b.offsets, b.perm_row,
                              inp["W_r"], st["dW_r"], st["dbias"], b.dX)
    return {"idx": b.idx, "gate": b.gate, "counts": b.counts, "Y": b.Y, "dX": b.dX, "dgate": b.dgate, "dW_gate": b.dW_gate,
            "dW_up": b.dW_up, "dW_down": b.dW_down, "dW_r": st["dW_r"], "dbias": st["dbias"]}


def _chunked_step(st):
    ctx, inp, C = st["ctx"], st["inp"], st["case"]["chunks"]
    weights = (inp["W_gate"], inp["W_up"], inp["W_down"])
    tables = (st["offsets"], st["perm_row"], st["row_src"])
    binding.mop_moe_layer_fwd_chunked(ctx, C, inp["x"], inp["W_r"], inp["bias"], *weights, st["idx"], st["gate"], st["counts"],
                                      *tables, st["Y"], st["ws"])
    binding.mop_moe_layer_bwd_chunked(ctx, C, inp["x"], inp["dY"], st["gate"], *tables, *weights, st["dX"], st["dW_gate"],
                                      st["dW_up"], st["dW_down"], st["dgate"], st["ws"])
    return {n: st[n] for n in ("idx", "gate", "counts", "Y", "dX", "dgate", "dW_gate", "dW_up", "dW_down")}


def run(state):
    case = state["case"]
    if case["pass"] == "fwd":
        b = state["buf"]
        binding.forward(state["ctx"], state["inp"], b)
        return {"idx": b.idx, "gate": b.gate, "counts": b.counts, "Y": b.Y}
    if case["pass"] == "train":
        return _train_step(state)
    if case["pass"] == "chunked":
        return _chunked_step(state)
    dev = state["X"].device.index
    binding.mop_vocab_loss_fwd(dev, state["X"], state["W"], state["targets"], state["loss"], state["lse"], state["ws"])
    if case["pass"] == "vocab_fwd":
        return {"loss": state["loss"], "lse": state["lse"]}
    binding.mop_vocab_loss_bwd(dev, state["X"], state["W"], state["targets"], state["lse"], state["dloss"], state["dX"],
                               state["dW"], state["ws_bwd"])
    return {"loss": state["loss"], "lse": state["lse"], "dX": state["dX"], "dW": state["dW"]}


def work(case):
    """Every input once, every output once, the products that the results need.  Weights: of the experts that get rows."""
    if case["pass"].startswith("vocab"):
        N, H, V = case["N"], case["H"], case["V"]
        if case["pass"] == "vocab_fwd":
            return {"bytes": 2 * N * H + 2 * H * V + 12 * N, "flops": 2 * N * H * V}
        return {"bytes": 4 * N * H + 6 * H * V + 16 * N, "flops": 6 * N * H * V}
    T, d, E, k, f = (case[n] for n in ("T", "d", "E", "k", "f"))
    M = T * k
    live = E - math.ceil(0.1 * E) if case["skew"] else E * (1.0 - (1.0 - k / E) ** T)
    nbytes = 4 * T * d + 4 * d * E + 6 * live * d * f + 8 * M
    flops = 6 * M * d * f + 2 * T * d * E
    if case["pass"] != "fwd":
        nbytes += 4 * T * d + 12 * E * d * f + 4 * M
        flops += 12 * M * d * f
    if case["pass"] == "train":
        nbytes += 4 * d * E
        flops += 4 * M * d
    return {"bytes": int(nbytes), "flops": int(flops)}


def tolerance(case):
    # Indices and counts are exact in every implementation (the routing contract fixes each logit's chain of additions).  The other
    # outputs are fp32 sums of bf16 products with intermediates rounded to bf16 in between; with the sums in another order an
    # intermediate flips to its neighbour now and then.  Seen against fp64 sums with the same roundings, at d = 512 to 7168
    # (2-norm; largest difference): bf16 outputs 3e-4 to 1.5e-3; 0.018, fp32 gradients 5e-5 to 3.3e-4; 0.032.  The vocabulary's loss
    # 2.3e-6; 5e-6 (fp32, nothing rounded to bf16), its dX 2.4e-4; 0.008 (one rounding of the logits' gradients).  Four times those.
    if case["pass"] == "vocab_fwd":
        return {"rel": 1e-5, "max": 2e-5}
    if case["pass"] == "vocab_train":
        return {"rel": 1e-3, "max": 0.032}
    return {"rel": 6e-3, "max": 0.12}
