"""The work a BranchGRPO training program has this library do, as timed cases.

A program of this library runs, per iteration, a *rollout pass* for every prompt batch (root latents, T denoising steps with
forks, leaf rewards, fused values and advantages, gradient masks), and while it updates the policy it *scores* the stored
trees again (log-probs under new velocities, clipped objective).  Around these stand the tree reductions on their own
(rewards that come from elsewhere, other settings tried on the same trees), and the reward call that brings its own scratch.

Kinds of case
  pass    one whole pass of ``TreeSession``: rollout, rewards, fusion and advantages, pruning
  score   log-probs of every stored edge under given velocities (or the bound closed form) and the clipped objective
  reduce  fusion with path weights, effective sample size, pruning, objective on finished trees
  static  ``reward_mse_static``: -MSE rewards of latent rows with the library's built-in scratch
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_06040_b200 import binding as B
from paper_2509_06040_b200.session import TreeSession
from workloads import (CONFIGS, WIDTH_EXTREME_B, WIDTH_LAST_SPLIT_TOPK, WIDTH_NONE, WIDTH_PER_SPLIT_TOPK, Workload,
                       make_inputs)

DEVICE = "cuda:0"

_DEFAULTS = dict(kind="pass", n_trees=1, tokens=16, channels=64, T=16, K=2, splits="0,3,6,9", sigma=0.3, velocity="mlp",
                 reward="mixture", hidden=3072, corr_s=0.0, beta=0.0, adv_clip=0.0, width_mode=WIDTH_NONE, width_k=0,
                 n_pruned=0, window=0, one_launch=False)


def _case(name=None, **kw):
    c = dict(_DEFAULTS)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def _of_config(name, kind="pass", **kw):
    """A case with the shape and schedule of one of the repository's named configurations."""
    w = CONFIGS[name]
    c = dict(kind=kind, n_trees=w.n_trees, tokens=w.tokens, channels=w.channels, T=w.T, K=w.K,
             splits=",".join(map(str, w.splits)), sigma=w.sigma, velocity=w.velocity, reward=w.reward, hidden=w.hidden,
             beta=w.beta, width_mode=w.width_mode, width_k=w.width_k, n_pruned=w.n_pruned_depths)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest program: one prompt of 16 x 4 elements, four steps.  Launches and host time only.
        _case("toy_pass", **_of_config("toy")),
        # A 256 x 256 image (16 x 16 patches), one prompt, the denoiser stand-in at full width: small launches of every kernel.
        _case("thumbnail_pass", n_trees=1, tokens=256, T=16, splits="0,3,6,9", reward="normal_plus_cos"),
        # One 720 x 720 image prompt: interactive use, one prompt at a time.
        _case("image_pass", **_of_config("image")),
        # The batch one GPU takes per iteration: 32 prompts, top-2 per split, pruned depths.
        _case("image_batch_pass", **_of_config("image_batch")),
        # The largest single-GPU configuration: 8 prompts of 1024 x 1024, 64 leaves each (the benchmark's default workload).
        _case("group_pass", **_of_config("group")),
        # Ragged sizes and the method's options together: odd token count, a narrower denoiser whose hidden width is no power
        # of two, K = 3 forks with correlated branch noise, hybrid ODE-SDE schedule, path-weighted fusion, clipped advantages,
        # Extreme-b pruning.
        _case("ragged_hybrid_pass", n_trees=3, tokens=1531, T=20, K=3, splits="0,4,9", hidden=1408, corr_s=2.0, window=6,
              reward="normal_plus_cos", beta=1.0, adv_clip=5.0, width_mode=WIDTH_EXTREME_B, width_k=4, n_pruned=2),
        # A video latent (21 x 60 x 104 x 16) with the closed-form velocity, step by step.
        _case("video_pass", **_of_config("video")),
        # A batch of image latents with the closed-form velocity in one launch (the entry point for launch-bound sizes).
        _case("one_launch_pass", n_trees=4, tokens=2025, velocity="linear", reward="neg_mse_target", one_launch=True,
              width_mode=WIDTH_PER_SPLIT_TOPK, width_k=1),
        # Policy update on image trees: every edge of four trees under a new policy's velocities, then the clipped objective.
        _case("image_score", **_of_config("image", kind="score", n_trees=4, width_mode=WIDTH_PER_SPLIT_TOPK, width_k=1)),
        # The same for a video tree under the bound closed form: all edges in one call.
        _case("video_score", **_of_config("video", kind="score")),
        # Reductions of 32 wide trees (K = 3, four splits, 81 leaves) with path weights: fusion, effective sample size, Parent-Top1
        # masks, objective.
        _case("wide_tree_reduce", kind="reduce", n_trees=32, tokens=16, channels=4, T=20, K=3, splits="0,3,6,9",
              velocity="linear", reward="mixture", beta=1.0, adv_clip=5.0, width_mode=WIDTH_LAST_SPLIT_TOPK, width_k=1, n_pruned=4),
        # Rewards of one image tree's 16 leaves from a caller without device scratch.
        _case("static_reward", kind="static", n_trees=16, tokens=2025),
    ]


# Largest drawn case: what the largest listed one (group_pass) writes and computes.
_MAX_POOL_BYTES = 6.4e9
_MAX_FLOPS = 1.8e13


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pass"] * 7 + ["score"] * 2 + ["reduce"] * 2 + ["static"])
    if kind == "static":      # rows within what the built-in scratch holds
        return _case(kind=kind, n_trees=_log_int(rng, 1, 64), tokens=_log_int(rng, 16, 4096))
    T = rng.randint(4, 20)
    K = rng.choice([2, 2, 2, 3, 4])
    most = {2: 6, 3: 4, 4: 3}[K]
    splits = sorted(rng.sample(range(max(1, (2 * T) // 3)), rng.randint(1, min(most, (2 * T) // 3))))
    c = _case(kind=kind, T=T, K=K, splits=",".join(map(str, splits)), sigma=rng.choice([0.3, 0.5]),
              corr_s=rng.choice([0.0, 0.0, 1.0, 2.0, 4.0]), beta=rng.choice([0.0, 0.0, 1.0]), adv_clip=rng.choice([0.0, 5.0]),
              n_trees=_log_int(rng, 1, 32))
    if kind == "pass":
        mode = rng.choice([WIDTH_NONE, WIDTH_PER_SPLIT_TOPK, WIDTH_LAST_SPLIT_TOPK, WIDTH_EXTREME_B])
        k = 0 if mode == WIDTH_NONE else rng.randint(1, 4 if mode == WIDTH_EXTREME_B else 2)
    else:                     # Parent-Top1: a mask that keeps whole sibling groups makes the objective a sum that cancels to zero
        mode, k = rng.choice([WIDTH_PER_SPLIT_TOPK, WIDTH_LAST_SPLIT_TOPK]), 1
    c.update(width_mode=mode, width_k=k, n_pruned=rng.choice([0, 0, 2, min(4, T - 1)]))
    if kind == "reduce":
        c.update(tokens=16, channels=4, velocity="linear", reward="mixture")
    elif rng.random() < 0.6:  # the denoiser stand-in
        c.update(velocity="mlp", tokens=_log_int(rng, 64, 4096), hidden=128 * _log_int(rng, 2, 24),
                 reward=rng.choice(["mixture", "normal_plus_cos"]), window=rng.choice([0, 0, 4]) if kind == "pass" else 0)
    else:                     # the closed form
        c.update(velocity="linear", channels=rng.choice([4, 16, 64]), reward=rng.choice(["neg_mse_mu", "neg_mse_target"]),
                 one_launch=kind == "pass" and rng.random() < 0.3)
        c["tokens"] = _log_int(rng, 16, 2_100_000 // c["channels"])
    while True:               # no larger than the largest listed case
        w = _workload(c, 0)
        pool = 4.0 * c["n_trees"] * w.nodes * w.D * (2 if kind == "score" else 1)
        if pool <= _MAX_POOL_BYTES and _mlp_flops(c, w) <= _MAX_FLOPS:
            return c
        if c["n_trees"] > 1:
            c["n_trees"] = (c["n_trees"] + 1) // 2
        else:
            c["tokens"] = (c["tokens"] + 1) // 2


def _splits(c):
    return tuple(int(x) for x in c["splits"].split(","))


def _workload(c, seed):
    return Workload(name="case", n_trees=c["n_trees"], tokens=c["tokens"], channels=c["channels"], T=c["T"], K=c["K"],
                    splits=_splits(c), sigma=c["sigma"], velocity=c["velocity"], reward=c["reward"], hidden=c["hidden"],
                    branch_corr_s=c["corr_s"] if c["corr_s"] > 0 else math.inf, beta=c["beta"], adv_clip=c["adv_clip"],
                    width_mode=c["width_mode"], width_k=c["width_k"], n_pruned_depths=c["n_pruned"], seed=1223627 + seed,
                    input_seed=42 + seed)


def prepare(case, seed):
    rng = torch.Generator(device=DEVICE).manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, device=DEVICE, generator=rng)

    if case["kind"] == "static":
        D = case["tokens"] * case["channels"]
        return {"case": case, "rows": normal(case["n_trees"], D), "target": normal(D),
                "r": torch.empty(case["n_trees"], device=DEVICE)}
    w = _workload(case, seed)
    s = TreeSession(w, device=DEVICE, fused_rollout=case["one_launch"])
    s.upload_inputs(make_inputs(w))
    state = {"case": case, "s": s}
    if case["window"]:        # hybrid schedule: the split steps and a window stay stochastic
        s.init()
        stochastic = B.mix_sde_steps(w.T, w.splits, iteration=60, window=case["window"], every=30, start=1)
        B.tree_set_sde_steps(s.tree, [1 if i in stochastic else 0 for i in range(w.T)])
    if case["kind"] == "pass":
        return state
    # finished trees, as the rollout left them
    s.run_all()
    state["terms"] = torch.empty_like(s.logp)
    state["J"] = torch.empty(w.n_trees, device=DEVICE)
    if case["kind"] == "score":
        state["logp_new"] = torch.zeros_like(s.logp)
        if w.velocity == "mlp":      # the new policy's velocities of every parent, step by step
            state["v"] = [0.1 * normal(w.n_trees, W, w.D) for W in w.widths()[:-1]]
    else:
        state["logp_new"] = s.logp + 1e-4 * normal(*s.logp.shape)
        state["ess"] = torch.empty_like(s.logp)
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "static":
        B.reward_mse_static(state["rows"], state["target"], case["n_trees"], case["tokens"] * case["channels"], state["r"])
        return {"r": state["r"]}
    s = state["s"]
    if case["kind"] == "pass":
        s.run_all()
        return {"latents": s.latents, "table": s.node_table, "logp": s.logp, "leaf_r": s.leaf_r, "rbar": s.rbar, "adv": s.adv,
                "mask": s.mask}
    if case["kind"] == "score":
        if "v" in state:
            for i, v in enumerate(state["v"]):
                B.tree_logprob(s.tree, i, v, state["logp_new"])
        else:
            B.tree_logprob(s.tree, -1, None, state["logp_new"])
        B.tree_grpo_objective(s.tree, state["logp_new"], logp_scale=1.0, clip_eps=1e-4, terms_out=state["terms"], J_out=state["J"])
        return {"logp_new": state["logp_new"], "terms": state["terms"], "J": state["J"]}
    s.fuse_advantage()
    B.tree_fusion_ess(s.tree, case["beta"], 1.0, state["ess"])
    s.prune()
    B.tree_grpo_objective(s.tree, state["logp_new"], logp_scale=1.0, clip_eps=1e-4, terms_out=state["terms"], J_out=state["J"])
    return {"rbar": s.rbar, "adv": s.adv, "ess": state["ess"], "mask": s.mask, "terms": state["terms"], "J": state["J"]}


def _mlp_flops(case, w):
    if w.velocity != "mlp" or case["kind"] != "pass":
        return 0.0
    return 4.0 * w.channels * w.hidden * w.tokens * w.model_evals * w.n_trees


def work(case):
    if case["kind"] == "static":
        n = case["tokens"] * case["channels"]
        return {"bytes": 4.0 * n * (case["n_trees"] + 1), "flops": 3.0 * n * case["n_trees"]}
    w = _workload(case, 0)
    rows, D = w.n_trees * w.nodes, w.D
    if case["kind"] == "reduce":     # logp in (fusion, ESS), logp_new in; rbar, adv, ess, terms, mask out
        return {"bytes": rows * (4 * 6 + 1) + 4.0 * w.n_trees * (w.leaves + 1), "flops": 40.0 * rows}
    edges = w.n_trees * w.node_steps
    if case["kind"] == "score":      # every stored latent once, every parent's velocity (or the target mean) once
        operand = w.n_trees * w.model_evals * D if w.velocity == "mlp" else w.n_trees * D
        return {"bytes": 4.0 * (rows * D + operand + 6 * rows), "flops": 6.0 * edges * D}
    # a pass writes every node's latent once and reads the target mean, the reward target and the weights once
    inputs = w.n_trees * D * ((w.velocity == "linear") + (w.reward in ("neg_mse_target", "normal_plus_cos")))
    weights = 4.0 * w.channels * w.hidden if w.velocity == "mlp" else 0.0
    return {"bytes": 4.0 * (rows * D + inputs) + weights + rows * (4 * 7 + 1) + 4.0 * w.n_trees * w.leaves,
            "flops": 6.0 * edges * D + _mlp_flops(case, w)}


def tolerance(case):
    # About four times what each path differs by from itself in 64 bits (float32 kept where the state format is float32).
    if case["velocity"] == "mlp" and case["kind"] == "pass":
        # bf16 activations inside the velocity: latents 6e-5 (worst element 4.4e-4); log-probs and values 2e-7
        return {"rel": 2.5e-4, "max": 2e-3}
    if case["velocity"] == "linear" and case["kind"] in ("pass", "score"):
        # latents and log-probs 2e-7; -MSE rewards of leaves are close to one another (spread ~ 1/sqrt(D)), so the float32
        # rounding of a reward shows in the advantages: 8.6e-5 (worst 2.5e-4) at 2 M elements
        return {"rel": 4e-4, "max": 1e-3}
    # float32 sums over a row, float32 results of double arithmetic: 1e-7 (worst 4e-6)
    return {"rel": 1e-5, "max": 4e-5}
