"""Performance cases: the calls that a reinforcement-learning trainer makes on this library, over the sizes,
types and options that it makes them with.

``listed()`` are fixed workloads, ``draw()`` gives further ones from the same ranges.  Inputs are the seeded
synthetic batches of ``paper_2512_23087_b200.inputs`` (logits with a few dominant tokens over a Gaussian or
heavy-tailed base, inference logits = training logits + noise, tokens sampled from the inference policy).
"""
from __future__ import annotations

import math

import torch

from paper_2512_23087_b200 import binding, inputs

PAPER_RHO = math.exp(-13.0)   # the threshold of the paper's experiments
_BYTES = {"f32": 4, "bf16": 2, "f16": 2}

# base, scale, head boost, most head tokens, sigma of infer - train: the generators of the repository's configurations
_SHAPES = {
    "small": ("normal", 3.0, 12.0, 8, 0.01),
    "peaked": ("normal", 3.0, 15.0, 8, 0.02),
    "heavy": ("student_t3", 4.0, 15.0, 16, 0.05),
}


def _rows(kind, T, V, dtype, rho, shape="peaked", **more):
    """A case over stored logits.  ``pad``: elements between the rows (0: contiguous); ``mask_value``: 0.0 for the
    exact -inf semantics, else the finite value that pruned logits take; ``keep_grad``: the program owns the
    gradient matrix and hands it to every call."""
    c = {"kind": kind, "T": T, "V": V, "dtype": dtype, "rho": rho, "shape": shape, "grad_dtype": dtype, "pad": 0,
         "mask_value": 0.0, "keep_grad": False}
    c.update(more)
    return c


def listed():
    return [
        # one gradient step on a toy vocabulary, as in unit-scale experiments: launch and host latency
        dict(_rows("train", 64, 4096, "f32", 1e-3, "small"), name="small_train_f32"),
        # scoring the newest tokens of a few rollouts at the paper's threshold, no gradient
        dict(_rows("forward", 16, 151936, "bf16", PAPER_RHO), name="few_tokens_forward_bf16"),
        # a micro-batch of one 512-token response, forward and gradient
        dict(_rows("train", 512, 151936, "bf16", 1e-4), name="one_response_train_bf16"),
        # an odd vocabulary whose rows lie back to back, so that no two rows are aligned alike
        dict(_rows("train", 1111, 50021, "f16", 1e-3), name="odd_vocab_train_f16"),
        # log-probabilities of a rollout batch under both policies (the old-policy pass)
        dict(_rows("forward", 8192, 151936, "bf16", 1e-4), name="rollout_forward_bf16"),
        # the training step over 64 responses of 512 tokens, gradient buffer owned by the trainer
        dict(_rows("train", 32768, 151936, "bf16", 1e-4, keep_grad=True), name="batch_train_bf16"),
        # float32 logits of a 262,144-token vocabulary with heavy tails
        dict(_rows("train", 4096, 262144, "f32", 1e-4, "heavy", keep_grad=True), name="heavy_train_f32"),
        # token-level truncated importance weights formed inside the call
        dict(_rows("weighted", 2048, 151936, "bf16", 1e-4), name="weighted_train_bf16"),
        # sequence-level weights: forward, aggregation over the responses, then the stand-alone backward
        dict(_rows("two_call", 4096, 151936, "bf16", PAPER_RHO), name="sequence_weights_bf16"),
        # divergence and entropy monitoring of the two policies
        dict(_rows("monitor", 4096, 151936, "bf16", 1e-4), name="monitor_bf16"),
        # LM head fused with the loss: a small model's micro-batch, and the full batch of a large one
        dict({"kind": "fused", "T": 512, "H": 1024, "V": 32000, "rho": 1e-4}, name="fused_small_model"),
        dict({"kind": "fused", "T": 16384, "H": 4096, "V": 151936, "rho": 1e-4}, name="fused_large_model"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "train", "train", "train", "weighted", "two_call", "monitor", "fused"])
    if kind == "fused":
        T, H, V = _log_int(rng, 32, 8192), 8 * _log_int(rng, 32, 512), _log_int(rng, 2000, 152000)
        T = max(32, min(T, int(2.5e12 / (H * V))))
        return {"kind": "fused", "T": T, "H": H, "V": V, "rho": rng.choice([1e-4, PAPER_RHO])}
    V = _log_int(rng, 2000, 262144)
    V = max(16, V // rng.choice([1, 1, 16, 64, 64]) * 64) if rng.random() < 0.5 else V   # half of them round sizes
    V = min(V, 262144)
    shape = rng.choice(["peaked", "peaked", "heavy"])
    # heavy-tailed rows put nearly all mass on one token: single log-probabilities then are the rounding of two nearly
    # equal sums, and only batches have results to compare
    T = max(1, min(_log_int(rng, 256 if shape == "heavy" else 4, 32768), int(1.2e9 / V)))
    rho = rng.choice([1e-4, 1e-3] if shape == "heavy" else [1e-4, 1e-3, PAPER_RHO])
    dtype = rng.choice(["bf16", "bf16", "f16", "f32"])
    more = {"pad": rng.choice([0, 0, 0, 16 - V % 16]), "mask_value": rng.choice([0.0, 0.0, 0.0, -50.0])}
    if kind in ("train", "two_call"):
        more["grad_dtype"] = rng.choice([dtype, dtype, "f32"])
    return _rows(kind, T, V, dtype, rho, shape, **more)


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "fused":
        w = inputs.FusedWorkload("lm_head", case["T"], case["H"], case["V"], 0.02, 0.02, (case["rho"],))
        return {"case": case, "batch": inputs.make_fused(w, seed=seed, device=dev)}
    base, scale, boost, heads, sigma = _SHAPES[case["shape"]]
    T, V = case["T"], case["V"]
    w = inputs.RowWorkload("rows", T, V, case["dtype"], base, scale, boost, heads, sigma, (case["rho"],), True)
    state = {"case": case, "batch": inputs.make_rows(w, seed=seed, device=dev, ld=V + case["pad"]), "grad": None}
    if case["keep_grad"]:
        state["grad"] = torch.zeros(T, V, dtype=inputs.torch_dtype(case["grad_dtype"]), device=dev)
    if case["kind"] == "two_call":   # responses of at most 512 tokens
        n = (T + 511) // 512
        state["offsets"] = torch.clamp(torch.arange(n + 1, device=dev) * 512, max=T)
        state["sequence_of"] = torch.arange(T, device=dev) // 512
        g = torch.Generator(device=dev)
        g.manual_seed(int(seed))
        state["advantage"] = torch.randn(n, generator=g, device=dev)
    return state


def _side(o, coverage=True):
    names = ("max", "lse", "lse_safe", "logp", "logp_mp", "comp_mp", "count") + (("log_cov",) if coverage else ())
    return {n: getattr(o, n) for n in names}


def run(state):
    c, b = state["case"], state["batch"]
    kind, rho = c["kind"], c["rho"]
    if kind == "fused":
        r = binding.dvp_fused_lmhead_forward_backward(b.hidden, b.w_vocab, b.ids, rho, b.upstream, infer_logits=b.infer)
        return {"train": _side(r.train), "infer": _side(r.infer), "log_ratio": r.log_ratio, "flags": r.flags,
                "d_hidden": r.d_hidden, "d_w": r.d_w}
    if kind == "monitor":
        r = binding.dvp_monitor(b.train, b.infer)
        return {"kl_infer_train": r.kl_infer_train, "kl_train_infer": r.kl_train_infer,
                "entropy_train": r.entropy_train, "entropy_infer": r.entropy_infer}
    mask_value = c["mask_value"] or None
    grad = {"grad_train": state["grad"], "grad_dtype": inputs.torch_dtype(c["grad_dtype"])}
    if kind == "forward":
        r = binding.dvp_forward(b.train, b.ids, rho, infer_logits=b.infer, mask_value=mask_value)
    elif kind == "train":
        r = binding.dvp_forward(b.train, b.ids, rho, infer_logits=b.infer, upstream=b.upstream, mask_value=mask_value,
                                **grad)
    elif kind == "weighted":
        r = binding.dvp_forward(b.train, b.ids, rho, infer_logits=b.infer, upstream=b.upstream, mask_value=mask_value,
                                weight_kind=binding.DVP_WEIGHT_TRUNCATE, weight_hi=1.2, **grad)
    else:
        r = binding.dvp_forward(b.train, b.ids, rho, infer_logits=b.infer, mask_value=mask_value)
        s = binding.dvp_sequence_aggregate(r.log_ratio, state["offsets"], log_cov=r.train.log_cov)
        weight = torch.exp(s.seq_log_ratio).clamp(max=1.2) * (1 - s.veto) * state["advantage"]
        upstream = weight[state["sequence_of"]]
        r.grad_train = binding.dvp_backward(b.train, b.ids, rho, upstream, r, mask_value=mask_value, **grad)
    # ln Z of a heavy-tailed row is 1e-5 and less, below the rounding of the two sums it is formed from
    coverage = c["shape"] != "heavy"
    out = {"train": _side(r.train, coverage), "infer": _side(r.infer, coverage), "log_ratio": r.log_ratio,
           "flags": r.flags, "grad_train": r.grad_train}
    if kind == "weighted":
        out["weight"] = r.weight
    if kind == "two_call":
        out["sequences"] = {"log_ratio": s.seq_log_ratio, "min": s.min_log_ratio, "valid": s.n_valid,
                            "zero": s.n_zero_weight, "veto": s.veto, "min_cov": s.min_cov, "mean_cov": s.mean_cov}
    return out


def work(case):
    T, V, kind = case["T"], case["V"], case["kind"]
    if kind == "fused":
        # logits, d_hidden and d_w: three contractions.  At these thresholds the generator's rows keep nearly every
        # token, so the gradient contractions have nothing to skip.  Hidden rows, weights and their float32 gradients
        # once, the inference logits once.
        H = case["H"]
        return {"flops": 6.0 * T * V * H, "bytes": 6.0 * (T + V) * H + 2.0 * T * V}
    z, g = _BYTES[case["dtype"]], _BYTES[case["grad_dtype"]]
    per_logit = {"forward": 2 * z, "monitor": 2 * z, "train": 2 * z + g, "weighted": 2 * z + g,
                 # every sequence's weight needs all of its tokens before any gradient: the training logits are an
                 # input of both calls
                 "two_call": 3 * z + g}[kind]
    # an exponential, a multiply-add, a comparison and an addition per logit and side
    return {"bytes": float(T) * V * per_logit + 100.0 * T, "flops": 10.0 * T * V}


def tolerance(case):
    """About four times the distance of every output from a float64 evaluation of the definitions (measured at up to
    1,200 tokens)."""
    if case["kind"] == "fused":
        # ln Z of the inference rows 1.7e-3; a logit within accumulation rounding of the threshold may fall either way
        return {"rel": 7e-3, "max": 2e-2, "differ": 1e-2}
    if case["kind"] == "monitor":   # a divergence of 2e-4 from sums of order one: 1.7e-3
        return {"rel": 7e-3, "max": 2.5e-2}
    if case["kind"] != "forward" and case["grad_dtype"] == "bf16":   # the rounding of the stored gradient: 1.7e-3
        return {"rel": 7e-3, "max": 1.6e-2}
    # ln Z 3.8e-4 where it is 1e-3, log-ratios 1.4e-4, float16 gradients 2.3e-4
    return {"rel": 1.5e-3, "max": 5.5e-3}
