"""What a user has the FGMP linear layer do, as cases that can be timed and compared.

Every case is one linear layer of a transformer (or the two of a feed-forward block) at the shapes that this repository's
configurations name, called through the package's public functions the way an inference program calls them: weights are
packed once and kept with their workspace, activations come in as bf16 and are quantized on the fly.

  decode   `linear_fused`: one decode step of a small batch (1 to 16 tokens)
  layer    `quantize_activations` + `linear`: any other batch -- many sequences decoding together, and prefill
  mlp      `quantize_activations` + `linear_quantize` + `linear`: both linears of a feed-forward block, the tensor between
           them in packed form only
  offline  `calibrate_tau` + `quantize_weights` + `unpack`: what preparing one layer for deployment takes -- the activation
           threshold from a calibration batch, the packed weights, and their canonical arrays for a checkpoint
"""
import math

import torch

import paper_2504_14152_b200 as fg
from paper_2504_14152_b200 import binding as fgb

DEV = "cuda"


def listed():
    return [
        # the repository's smallest configuration: all fixed cost
        dict(name="tiny-m64", kind="layer", M=64, N=256, K=256, fp8=0.10, out="fp32", score=0),
        # one user's decode step on the widest linear of a 7B model: latency
        dict(name="decode-7b-fc1-m1", kind="decode", M=1, N=11008, K=4096, fp8=0.10, out="bf16", score=0),
        # the benchmark's default workload
        dict(name="decode-7b-fc1-m16", kind="decode", M=16, N=11008, K=4096, fp8=0.10, out="fp32", score=0),
        # a ragged decode batch on the long-K projection of a 13B model, ranked with the other block score
        dict(name="decode-13b-fc2-m7", kind="decode", M=7, N=5120, K=13824, fp8=0.10, out="bf16", score=1),
        # the largest decode weights: bound by the weight stream
        dict(name="decode-70b-fc1-m1", kind="decode", M=1, N=28672, K=8192, fp8=0.10, out="bf16", score=0),
        # continuous batching: more sequences than the decode kernel takes
        dict(name="batch-7b-o-m48", kind="layer", M=48, N=4096, K=4096, fp8=0.10, out="bf16", score=0),
        # a short prompt, or a chunk of a prefill, at a ragged length
        dict(name="batch-13b-fc1-m203", kind="layer", M=203, N=13824, K=5120, fp8=0.20, out="bf16", score=0),
        # the paper's prefill: a 7B layer at 4096 tokens
        dict(name="prefill-7b-fc1-m4096", kind="layer", M=4096, N=11008, K=4096, fp8=0.10, out="bf16", score=0),
        # the all-NVFP4 end of the FP8-fraction sweep
        dict(name="prefill-13b-fc1-nvfp4", kind="layer", M=2048, N=13824, K=5120, fp8=0.0, out="fp32", score=0),
        # the largest: a 70B layer at 8192 tokens
        dict(name="prefill-70b-fc1-m8192", kind="layer", M=8192, N=28672, K=8192, fp8=0.10, out="bf16", score=0),
        # a feed-forward block on a prompt of odd length
        dict(name="mlp-7b-m777", kind="mlp", M=777, N=11008, K=4096, fp8=0.10, out="bf16", score=0),
        # preparing one attention projection of a 7B model
        dict(name="offline-7b-o", kind="offline", M=512, N=4096, K=4096, fp8=0.10, clip=1, score=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "layer", "layer", "layer", "layer", "mlp", "offline"])
    # model widths are multiples of 256 nearly always; K % 64 == 0 is what the layer asks for, and N may be anything
    K = 256 * _log_int(rng, 1, 56) if rng.random() < 0.8 else 64 * _log_int(rng, 3, 200)
    N = 64 * _log_int(rng, 4, 224) if rng.random() < 0.7 else _log_int(rng, 250, 14336)
    fp8 = rng.choice([0.0, 0.05, 0.1, 0.1, 0.2, 0.3])
    out = rng.choice(["bf16", "bf16", "fp32"])
    score = rng.choice([0, 0, 1])
    if kind == "decode":
        K = 256 * max(1, K // 256)
        return dict(kind=kind, M=_log_int(rng, 1, 16), N=N, K=K, fp8=fp8, out=out, score=score)
    if kind == "layer":
        return dict(kind=kind, M=_log_int(rng, 17, 4096), N=N, K=K, fp8=fp8, out=out, score=score)
    if kind == "mlp":
        return dict(kind=kind, M=_log_int(rng, 17, 2048), N=64 * max(4, N // 64), K=K, fp8=fp8, out=out, score=score)
    return dict(kind=kind, M=_log_int(rng, 64, 2048), N=N, K=K, fp8=fp8, clip=rng.choice([0, 1, 1]), score=score)


# ---------------------------------------------------------------------------- inputs
# The distributions of the repository's seeded inputs (Llama-shaped: N(0, 1) activations with 1 % of the channels 30 times
# as large, N(0, 0.02) weights, log-normal Fisher information), drawn on the GPU.

def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000 + stream)
    return g


def _channels(K, seed):
    """Per input channel: the magnitude of its activations, and its Fisher information."""
    n_out = max(1, round(0.01 * K))
    gain = torch.ones(K, device=DEV)
    gain[torch.randperm(K, generator=_gen(seed, 1), device=DEV)[:n_out]] = 30.0
    fisher = torch.exp(torch.randn(K, generator=_gen(seed, 2), device=DEV) * 1.5)
    return gain, fisher


def _acts(M, gain, seed, stream):
    return (torch.randn(M, gain.numel(), generator=_gen(seed, stream), device=DEV) * gain).to(torch.bfloat16)


def _weights(N, K, seed, stream):
    w = (torch.randn(N, K, generator=_gen(seed, stream), device=DEV) * 0.02).to(torch.bfloat16)
    f = torch.randn(N, K, generator=_gen(seed, stream + 1), device=DEV).mul_(1.5).exp_()
    return w, f


def _scale(x):
    return float(x.abs().max()) / 2688.0


def _threshold(x, fisher, s4, case):
    if case["fp8"] == 0.0:
        return math.inf
    return float(fg.calibrate_tau(x, fisher, scale_fp4=s4, fp8_fraction=case["fp8"], score_mode=case["score"]))


def _pack(N, K, seed, stream, case):
    w, f = _weights(N, K, seed, stream)
    return fg.quantize_weights(w, f, fp8_fraction=case["fp8"], score_mode=case["score"])


def prepare(case, seed):
    kind, M, N, K = case["kind"], case["M"], case["N"], case["K"]
    gain, fisher = _channels(K, seed)
    s = {"kind": kind, "fisher": fisher, "score": case["score"]}
    if kind == "offline":
        s["x"] = _acts(M, gain, seed, 3)
        s["w"], s["fw"] = _weights(N, K, seed, 5)
        s["s4"], s["fp8"], s["clip"] = _scale(s["x"]), case["fp8"], case["clip"]
        return s
    cal = _acts(256, gain, seed, 3)          # the calibration batch fixes the tensor scale and the threshold
    s["s4"] = _scale(cal)
    s["tau"] = _threshold(cal, fisher, s["s4"], case)
    s["x"] = _acts(M, gain, seed, 4)
    s["w"] = _pack(N, K, seed, 5, case)
    s["dtype"] = torch.bfloat16 if case["out"] == "bf16" else torch.float32
    if kind == "mlp":
        s["w2"] = _pack(K, N, seed, 7, case)
        hidden = fg.linear(fg.quantize_activations(cal, fisher, scale_fp4=s["s4"], tau=s["tau"], score_mode=s["score"]),
                           s["w"], out_dtype=torch.bfloat16)
        _, s["fisher2"] = _channels(N, seed + 500_000)
        s["s4_2"] = _scale(hidden)
        s["tau2"] = _threshold(hidden, s["fisher2"], s["s4_2"], case)
        s["ws"] = fgb.alloc_workspace(fgb.OP_LINEAR_QUANTIZE, M, N, K, DEV)
        s["ws2"] = fgb.alloc_workspace(fgb.OP_LINEAR, M, K, N, DEV)
    else:
        s["ws"] = fgb.alloc_workspace(fgb.OP_LINEAR_FUSED if kind == "decode" else fgb.OP_LINEAR, M, N, K, DEV)
    return s


def run(s):
    if s["kind"] == "decode":
        return fg.linear_fused(s["x"], s["fisher"], s["w"], scale_fp4=s["s4"], tau=s["tau"], score_mode=s["score"],
                               out_dtype=s["dtype"], workspace=s["ws"])
    if s["kind"] == "layer":
        acts = fg.quantize_activations(s["x"], s["fisher"], scale_fp4=s["s4"], tau=s["tau"], score_mode=s["score"])
        return fg.linear(acts, s["w"], out_dtype=s["dtype"], workspace=s["ws"])
    if s["kind"] == "mlp":
        acts = fg.quantize_activations(s["x"], s["fisher"], scale_fp4=s["s4"], tau=s["tau"], score_mode=s["score"])
        hidden = fg.linear_quantize(acts, s["w"], s["fisher2"], scale_fp4=s["s4_2"], tau=s["tau2"], score_mode=s["score"],
                                    workspace=s["ws"])
        return fg.linear(hidden, s["w2"], out_dtype=s["dtype"], workspace=s["ws2"])
    tau = fg.calibrate_tau(s["x"], s["fisher"], scale_fp4=s["s4"], fp8_fraction=s["fp8"], score_mode=s["score"])
    packed = fg.quantize_weights(s["w"], s["fw"], fp8_fraction=s["fp8"], score_mode=s["score"], clip_mode=s["clip"])
    codes4, codes8, scales, mask = fg.unpack(packed)
    return {"tau": tau, "codes4": codes4, "codes8": codes8, "scales": scales, "mask": mask}


def _packed_bytes(rows, K, fp8):
    """The packed form by the format alone: 9 bytes for an NVFP4 block, 16 for an FP8 block, one mask bit each."""
    blocks = rows * K / 16
    return blocks * ((1 - fp8) * 9 + fp8 * 16 + 0.125)


def work(case):
    kind, M, N, K, fp8 = case["kind"], case["M"], case["N"], case["K"], case["fp8"]
    if kind == "offline":
        # activations and their Fisher vector, weights and their Fisher matrix in; canonical arrays out.  The search rounds
        # every weight under 126 scales (8 operations each) where it is asked for.
        out = N * K * (0.5 + 1 + 1 / 16 + 1 / 128) + 4
        return {"bytes": M * K * 2 + K * 4 + N * K * 6 + out, "flops": N * K * 8.0 * (126 if case["clip"] else 1) + M * K * 8.0}
    y = 2 if case["out"] == "bf16" else 4
    b = M * K * 2 + K * 4 + _packed_bytes(N, K, fp8)
    if kind == "mlp":
        return {"bytes": b + N * 4 + _packed_bytes(K, N, fp8) + M * K * y, "flops": 4.0 * M * N * K}
    return {"bytes": b + M * N * y, "flops": 2.0 * M * N * K}


def tolerance(case):
    if case["kind"] == "offline":
        return "exact"                       # codes, scales, masks and ranks are defined bit for bit
    if case["kind"] == "mlp":
        # the tensor between the linears is rounded to bf16 and to 4 or 8 bits: a sum taken in another order moves a few
        # of its values by a step
        return {"rel": 1e-2, "max": 5e-2}
    if case["out"] == "bf16":
        return {"rel": 4e-3, "max": 1e-2}
    return {"rel": 1e-5, "max": 2e-4}        # exact products, fp32 sums
