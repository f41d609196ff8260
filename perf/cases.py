"""Timed cases of the library: what its users run, at the sizes and in the forms they run it.

A case is one call sequence of one entry point on K gradients of D parameters:

  filter    gaf_filter_accumulate (Algorithm 1 + Eq. 5), the library's own choice of schedule
  anyseed   gaf_filter_accumulate_any_seed (the order-indifferent variant)
  bucketed  gaf_filter_accumulate_bucketed on S buckets
  stream    gaf_stream_begin, K - 1 x gaf_stream_push, gaf_stream_end
  pairwise  gaf_pairwise_cosdist
  cosdist   gaf_cosdist of two gradients

Outputs and workspace are allocated once and kept, as a training loop keeps them; every pass overwrites all outputs.
Inputs are the synthetic micro-gradients of ``workloads`` (``config``: one of the five named configurations drawn from
the seed; 0: the mixture model with rho ~ U(-0.2, 0.6), the range of configuration 2).
"""
import math

import numpy as np
import torch

import paper_2412_18052_b200 as gaf
from paper_2412_18052_b200 import workloads

RESNET18 = workloads.RESNET18_100_NUMEL
GPT2 = workloads.GPT2_SMALL_NUMEL


def _case(op, K, D, dtype, tau=0.97, config=0, stacked=False, S=0, name=None):
    case = {"op": op, "K": K, "D": D, "dtype": dtype, "tau": tau, "config": config, "stacked": stacked, "S": S}
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest calls: the gradient of one layer or of an adapter; the call itself is most of the cost
        _case("filter", 3, 65_537, "bf16", name="filter_k3_bf16_65k"),
        # a small network (configuration 1)
        _case("filter", 4, 1_000_000, "f32", config=1, name="filter_k4_f32_1m"),
        # two micro-gradients, the setting of the paper's experiments, on a ResNet18-sized network
        _case("filter", 2, RESNET18, "f32", name="filter_k2_f32_resnet18"),
        # a ResNet18-sized network with its tensors' scales (configuration 2)
        _case("filter", 4, RESNET18, "f32", config=2, name="filter_k4_f32_resnet18"),
        # a GPT-2-small-sized network, late in training: nearly orthogonal gradients (configuration 4)
        _case("filter", 8, GPT2, "f32", config=4, name="filter_k8_f32_gpt2"),
        # the largest: a billion bf16 parameters (configuration 5)
        _case("filter", 8, 1_000_000_000, "bf16", config=5, name="filter_k8_bf16_1g"),
        # many micro-gradients: one per worker of a larger data-parallel job
        _case("filter", 16, RESNET18, "f32", name="filter_k16_f32_resnet18"),
        # one decision per tensor of the network
        _case("bucketed", 4, RESNET18, "f32", config=2, S=62, name="bucketed_k4_f32_resnet18"),
        # micro-gradients that arrive one at a time
        _case("stream", 4, RESNET18, "f32", config=2, name="stream_k4_f32_resnet18"),
        # the distance matrix that the paper's figures track (configuration 3), gathered into one matrix
        _case("pairwise", 32, RESNET18, "bf16", config=3, stacked=True, name="pairwise_k32_bf16_resnet18"),
        # the same analysis on binary32 gradients of a smaller network, separate buffers, ragged length
        _case("pairwise", 24, 3_000_001, "f32", name="pairwise_k24_f32_3m"),
        # distance of two gradients, logged during training
        _case("cosdist", 2, RESNET18, "f32", config=2, name="cosdist_f32_resnet18"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["filter", "filter", "filter", "filter", "anyseed", "bucketed", "stream", "pairwise", "pairwise",
                     "cosdist"])
    dtype = rng.choice(["f32", "bf16"])
    K = 2 if op == "cosdist" else _log_int(rng, 2, {"bucketed": 8, "stream": 12}.get(op, 64))
    # 2 GB of gradients at most for the draws: the largest listed case has 16 GB
    most = 2_000_000_000 // (K * (4 if dtype == "f32" else 2))
    D = _log_int(rng, 10_000, min(most, 250_000_000))
    if rng.random() < 0.3:
        D = max(8, D // 1024 * 1024)            # lengths that are whole tiles, beside odd ones
    return _case(op, K, D, dtype, tau=rng.choice([0.9, 0.95, 0.97, 1.0]), stacked=rng.random() < 0.5,
                 S=_log_int(rng, 1, 256) if op == "bucketed" else 0)


def _offsets(case):
    """Bucket offsets: the 62 tensors of the ResNet18 layout where the length is that network's, else S buckets of
    very different lengths (lognormal shares), multiples of 8 elements."""
    D, S = case["D"], case["S"]
    if D == RESNET18 and S == 62:
        return [0] + [int(o) for o in np.cumsum(workloads.resnet18_tensor_sizes(100))]
    share = np.random.RandomState(S).lognormal(0.0, 1.5, S)
    cut = (np.cumsum(share / share.sum())[:-1] * D).astype(np.int64) // 8 * 8
    return [0] + [int(c) for c in cut] + [D]


def prepare(case, seed):
    K, D, dtype = case["K"], case["D"], case["dtype"]
    if case["config"]:
        w = workloads.config(case["config"], device="cuda", K=K, D=D, seed=seed % (1 << 31), stacked=case["stacked"])
    else:
        rho = np.random.RandomState(seed % (1 << 31)).uniform(-0.2, 0.6, size=K).tolist()
        w = workloads.mixture(K, D, dtype, rho, seed, device="cuda", stacked=case["stacked"])
    state = {"op": case["op"], "grads": w.grads, "tau": case["tau"],
             "ws": gaf.new_workspace(K, D, gaf.GAF_F32 if dtype == "f32" else gaf.GAF_BF16, device="cuda")}
    if case["op"] == "filter":
        state["out"] = {"macro_out": torch.empty(D, dtype=torch.float32, device="cuda"),
                        "mask_out": torch.empty(K, dtype=torch.uint8, device="cuda"),
                        "dist_out": torch.empty(K, dtype=torch.float32, device="cuda"),
                        "count_out": torch.empty(1, dtype=torch.int32, device="cuda")}
    elif case["op"] == "pairwise":
        state["out"] = {"dist_out": torch.empty(K, K, dtype=torch.float32, device="cuda"),
                        "gram_out": torch.empty(K, K, dtype=torch.float64, device="cuda")}
    elif case["op"] == "cosdist":
        state["out"] = {"dist_out": torch.empty(1, dtype=torch.float32, device="cuda"),
                        "stats_out": torch.empty(3, dtype=torch.float64, device="cuda")}
    else:
        state["macro"] = torch.empty(D, dtype=torch.float32, device="cuda")
    if case["op"] == "bucketed":
        state["offsets"] = _offsets(case)
    return state


def run(state):
    op, g, ws, tau = state["op"], state["grads"], state["ws"], state["tau"]
    if op == "filter":
        return gaf.gaf_filter_accumulate(g, tau, ws, **state["out"])
    if op == "anyseed":
        return gaf.gaf_filter_accumulate_any_seed(g, tau, ws, macro_out=state["macro"])
    if op == "bucketed":
        return gaf.gaf_filter_accumulate_bucketed(g, tau, state["offsets"], ws, macro_out=state["macro"])
    if op == "pairwise":
        return gaf.gaf_pairwise_cosdist(g, ws, **state["out"])
    if op == "cosdist":
        return gaf.gaf_cosdist(g[0], g[1], ws, **state["out"])
    gaf.gaf_stream_begin(g[0], state["macro"], ws)
    for t in range(1, len(g)):
        gaf.gaf_stream_push(g[t], t, tau, state["macro"], ws)
    return (state["macro"],) + gaf.gaf_stream_end(len(g), state["macro"], ws)


def work(case):
    """Every gradient read once, the macro-gradient written once; the K (K + 1) / 2 dot products that the decisions
    or the matrix rest on (two operations a product), the triple of a distance."""
    K, D, b = case["K"], case["D"], 4 if case["dtype"] == "f32" else 2
    if case["op"] == "cosdist":
        return {"bytes": 2 * b * D, "flops": 6 * D}
    out = 0 if case["op"] == "pairwise" else 4 * D
    return {"bytes": K * b * D + out, "flops": K * (K + 1) * D}


def tolerance(case):
    """Both input types give binary32 results of sums that are carried in binary32 at the lowest level.  Measured
    against the same arithmetic in binary64 over the listed cases and 14 drawn ones: relative error of the
    macro-gradient up to 9e-8, of distances up to 1.3e-7, of the Gram matrix up to 6.6e-7 (32 bfloat16 gradients);
    largest single difference 9.5e-7.  Four times that.  A decision that differs is an error."""
    return {"rel": 2.6e-6, "max": 3.8e-6, "differ": 0.0}
