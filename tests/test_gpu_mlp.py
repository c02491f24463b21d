"""The tcgen05 MLP velocity stage against the oracle's bf16-emulating MLP, stage by stage: at every depth the
oracle's frontier latents are written into the device pool (so both sides see the same z), the CUDA stage runs
through the C ABI, and its output is compared under  |d| <= 2e-2 |v| + 2e-2 rms(v)  and, on outputs of at least rms size,
under the plain relative bound 2e-2 (bf16 operands, fp32 accumulation; the CUDA side evaluates the erf-form GELU by a
polynomial for its even half in packed bf16 on |x| < 1 and by the tanh form on the hardware tanh outside).  The tree is then advanced with the oracle's velocity, so
later depths exercise frontiers of several nodes, several trees and ragged 128-token tiles."""
import math

import numpy as np
import pytest
import torch

from oracle import mlp, sde
from oracle import tree as otree
from workloads import Workload, make_inputs

from test_gpu_parity import B, LATENT_TOL, f32  # noqa: F401

pytestmark = pytest.mark.gpu


def _mlp_close(got, ref):
    """The stated bound |d| <= 2e-2 |v| + 2e-2 rms(v) on every output, and the plain relative bound |d| <= 2e-2 |v| on
    the outputs that are not small (|v| >= rms(v)), where the rms term would otherwise hide the error."""
    rms = float(np.sqrt(np.mean(ref.astype(np.float64) ** 2)))
    d = np.abs(got - ref)
    ok = bool(np.all(d <= 2e-2 * np.abs(ref) + 2e-2 * rms))
    large = np.abs(ref) >= rms
    if large.any():
        ok = ok and bool(np.all(d[large] <= 2e-2 * np.abs(ref[large])))
    return ok, float(d.max()), rms


@pytest.mark.parametrize("tokens,hidden,n_trees,K,splits", [(200, 256, 2, 2, (0, 2)), (37, 128, 3, 3, (1,)), (512, 3072, 1, 2, (0, 1))])
def test_mlp_stage_matches_oracle_at_every_depth(B, tokens, hidden, n_trees, K, splits):
    from paper_2509_06040_b200.session import TreeSession
    w = Workload(name="mlp", n_trees=n_trees, tokens=tokens, channels=64, T=3, K=K, splits=splits, sigma=0.3,
                 velocity="mlp", reward="mixture", hidden=hidden)
    inp = make_inputs(w)
    topo = otree.build_topology(w.T, w.K, w.splits)
    grid = w.t_grid().astype(np.float64)
    v_store = {}

    def vel_factory(t):
        def vel(z, i, p):
            v = mlp.mlp_velocity(z.reshape(w.tokens, w.channels), inp.W1, inp.W2).reshape(-1)
            v_store[(t, i, p)] = v
            return v
        return vel

    lats = [sde.rollout(topo, w.D, grid, f32(w.sigma), w.branch_corr_s, w.seed, vel_factory(t), tree_id=t, nodes_cap=topo.nodes)[0]
            for t in range(n_trees)]
    s = TreeSession(w)
    s.upload_inputs(inp)
    s.init()
    worst = 0.0
    for i in range(w.T):
        level = list(topo.level(i))
        for t in range(n_trees):       # same z on both sides: the oracle's frontier goes into the pool
            s.latents[t, level[0]:level[-1] + 1].copy_(torch.from_numpy(lats[t][level[0]:level[-1] + 1]))
        s.v.fill_(float("nan"))
        B.velocity_mlp(s.tree, s.packed, w.hidden, s.v)
        torch.cuda.synchronize()
        B.tree_sync_status(s.tree)
        ref = np.stack([np.stack([v_store[(t, i, p)] for p in level]) for t in range(n_trees)])
        got = s.v.cpu().numpy().reshape(-1)[:ref.size].reshape(ref.shape)
        ok, err, rms = _mlp_close(got, ref)
        assert ok, (i, err, rms)
        worst = max(worst, err / rms)
        B.tree_step(s.tree, 1 if i in w.splits else 0, torch.from_numpy(ref).cuda())
    torch.cuda.synchronize()
    print("worst |d| / rms(v) over the depths:", worst)
    assert worst < 2e-2
    # the teacher-forced steps reproduce the oracle's latents
    for t in range(n_trees):
        assert np.abs(s.latents[t].cpu().numpy() - lats[t]).max() <= LATENT_TOL


def test_mlp_special_weights(B):
    """Zero weights give v = 0; W1 = [I, -I], W2 = [I; -I] gives v = GELU(z) - GELU(-z) = z up to bf16 rounding."""
    from paper_2509_06040_b200.session import TreeSession
    from workloads import Inputs
    w = Workload(name="mlp_id", n_trees=1, tokens=130, channels=64, T=1, K=1, splits=(), sigma=0.3,
                 velocity="mlp", reward="mixture", hidden=128)
    W1 = np.concatenate([np.eye(64), -np.eye(64)], axis=1).astype(np.float32)
    W2 = np.concatenate([np.eye(64), -np.eye(64)], axis=0).astype(np.float32)
    for scale in (1.0, 0.0):
        s = TreeSession(w)
        s.upload_inputs(Inputs(W1=W1 * scale, W2=W2 * scale))
        s.init()
        B.velocity_mlp(s.tree, s.packed, w.hidden, s.v)
        torch.cuda.synchronize()
        z = s.latents[0, 0].cpu().numpy().reshape(130, 64)
        v = s.v.cpu().numpy().reshape(-1)[:130 * 64].reshape(130, 64)
        if scale == 0.0:
            assert np.all(v == 0.0)
        else:
            assert np.allclose(v, z, rtol=2 ** -6, atol=4e-3)


@pytest.mark.parametrize("w1_std", [0.03, 0.12, 0.5])
def test_mlp_activation_inside_and_outside_the_polynomial_range(B, w1_std):
    """Hidden pre-activations of standard deviation about 0.25, 1 and 4: threads whose 64 values all lie inside |x| < 1
    take the packed polynomial, the others the hardware-tanh form; both against the oracle's erf-GELU MLP."""
    from paper_2509_06040_b200.session import TreeSession
    from workloads import Inputs, _to_bf16_values
    w = Workload(name="mlp_range", n_trees=1, tokens=300, channels=64, T=1, K=1, splits=(), sigma=0.3,
                 velocity="mlp", reward="mixture", hidden=256)
    g = np.random.default_rng([3, int(w1_std * 100)])
    W1 = _to_bf16_values(w1_std * g.standard_normal((64, 256), dtype=np.float32))
    W2 = _to_bf16_values(0.02 * g.standard_normal((256, 64), dtype=np.float32))
    s = TreeSession(w)
    s.upload_inputs(Inputs(W1=W1, W2=W2))
    s.init()
    B.velocity_mlp(s.tree, s.packed, w.hidden, s.v)
    torch.cuda.synchronize()
    B.tree_sync_status(s.tree)
    z = s.latents[0, 0].cpu().numpy().reshape(300, 64)
    h = mlp.bf16_round(z).astype(np.float64) @ W1.astype(np.float64)
    inside = float(np.mean(np.abs(h) < 1.0))
    ref = mlp.mlp_velocity(z, W1, W2)
    got = s.v.cpu().numpy().reshape(-1)[:ref.size].reshape(ref.shape)
    ok, err, rms = _mlp_close(got, ref)
    print(f"w1_std {w1_std}: {inside:.3f} of the pre-activations inside the range, worst |d|/rms(v) = {err / rms:.4f}")
    assert ok, (err, rms)


def test_full_mlp_rollout_stays_close_to_the_oracle(B):
    """End to end with the CUDA MLP feeding the CUDA step: drift against the all-oracle rollout is reported, and
    bounded loosely (the 1e-5 latent tolerance cannot hold downstream of a bf16 stage)."""
    from paper_2509_06040_b200.session import TreeSession
    w = Workload(name="mlp_e2e", n_trees=1, tokens=256, channels=64, T=6, K=2, splits=(0, 3), sigma=0.3,
                 velocity="mlp", reward="mixture", hidden=512)
    inp = make_inputs(w)
    topo = otree.build_topology(w.T, w.K, w.splits)
    grid = w.t_grid().astype(np.float64)
    lat, logp = sde.rollout(topo, w.D, grid, f32(w.sigma), math.inf, w.seed,
                            lambda z, i, p: mlp.mlp_velocity(z.reshape(w.tokens, 64), inp.W1, inp.W2).reshape(-1))
    s = TreeSession(w)
    s.upload_inputs(inp)
    s.rollout()
    torch.cuda.synchronize()
    B.tree_sync_status(s.tree)
    drift = np.abs(s.latents[0].cpu().numpy() - lat).max()
    print("max latent drift through the bf16 stage:", drift)
    assert drift < 5e-3
    assert np.abs(s.logp[0].cpu().numpy() - logp).max() < 1e-3


def test_small_frontier_split_is_reproducible_and_agrees_with_the_unsplit_kernel(B):
    """A frontier of fewer tiles than SMs is also cut along the hidden dimension (several CTAs per tile, partial tiles
    added in a fixed order).  Two launches give identical bits, and the values agree with the same tree evaluated inside
    a batch large enough that no split happens (float32 sums in another order: a few ulps)."""
    from paper_2509_06040_b200.session import TreeSession
    small = Workload(name="mlp_small", n_trees=1, tokens=300, channels=64, T=2, K=2, splits=(0,), sigma=0.3,
                     velocity="mlp", reward="mixture", hidden=1024)
    big = small.scaled(n_trees=64)            # 64 x 3 tiles: more tiles than SMs, one CTA per tile
    inp_s, inp_b = make_inputs(small), make_inputs(big)
    a = TreeSession(small)
    a.upload_inputs(inp_s)
    a.init()
    b = TreeSession(big)
    b.upload_inputs(inp_b)
    b.init()
    torch.cuda.synchronize()
    assert torch.equal(a.latents[0, 0], b.latents[0, 0])            # tree 0 draws the same root in both
    outs = []
    for _ in range(2):
        a.v.fill_(float("nan"))
        B.velocity_mlp(a.tree, a.packed, small.hidden, a.v)
        torch.cuda.synchronize()
        outs.append(a.v.view(-1)[:small.D].clone())
    B.velocity_mlp(b.tree, b.packed, big.hidden, b.v)
    torch.cuda.synchronize()
    B.tree_sync_status(a.tree)
    B.tree_sync_status(b.tree)
    assert torch.equal(outs[0], outs[1])
    ref = b.v.view(-1)[:small.D]
    rms = ref.pow(2).mean().sqrt().item()
    assert (outs[0] - ref).abs().max().item() <= 1e-5 * rms + 1e-6 * ref.abs().max().item()


def test_repeated_passes_are_bit_identical(B):
    """The whole path twice with the same seed, and once more after a pass with another seed in between: every output
    is identical bit for bit.  Sums are taken in fixed orders and kernels that overlap on the stream (programmatic
    dependent launch, the split of small MLP frontiers) wait for what they depend on."""
    from paper_2509_06040_b200.session import TreeSession
    w = Workload(name="mlp_repeat", n_trees=2, tokens=333, channels=64, T=6, K=2, splits=(0, 2, 3), sigma=0.3,
                 velocity="mlp", reward="normal_plus_cos", hidden=512, width_mode=1, width_k=1)
    inp = make_inputs(w)
    s = TreeSession(w)
    s.upload_inputs(inp)

    def snapshot(seed):
        s.run_all(seed=seed)
        torch.cuda.synchronize()
        B.tree_sync_status(s.tree)
        return [t.clone() for t in (s.latents, s.logp, s.rbar, s.adv, s.mask, s.node_table, s.leaf_r)]

    first = snapshot(11)
    second = snapshot(11)
    other = snapshot(12)
    third = snapshot(11)
    for a, b, c in zip(first, second, third):
        assert torch.equal(a, b) and torch.equal(a, c)
    assert not torch.equal(first[0], other[0])


@pytest.mark.parametrize("chunks", [2, 3, 4, 5, 6, 7, 8, 9, 11, 24])      # clusters of 2, 3, 4, 5, 6, 7, 8, 3, none, 8 CTAs a tile
def test_every_cluster_size_agrees_with_the_unsplit_kernel(B, chunks):
    """Two tiles, the second one of two tokens, cut along the hidden dimension into each size of cluster there is; the
    reference is the same tree inside a batch of 82 tiles, which is not cut (float32 sums in another order)."""
    from paper_2509_06040_b200.session import TreeSession
    small = Workload(name="mlp_cluster", n_trees=1, tokens=130, channels=64, T=1, K=1, splits=(), sigma=0.3,
                     velocity="mlp", reward="mixture", hidden=128 * chunks)
    outs = []
    for w in (small, small, small.scaled(n_trees=80)):
        s = TreeSession(w)
        s.upload_inputs(make_inputs(w))
        s.init()
        s.v.fill_(float("nan"))
        B.velocity_mlp(s.tree, s.packed, w.hidden, s.v)
        B.tree_sync_status(s.tree)
        outs.append(s.v.view(-1)[:small.D].clone())
    assert torch.equal(outs[0], outs[1])
    # either side rounds a running float32 sum 8 times a chunk (one MMA per 16 hidden units), by at most 2^-23 of its value;
    # a running sum does not get past twice the largest output
    bound = 2 * (8 * chunks) * 2.0 ** -23 * 2 * outs[2].abs().max().item()
    err = (outs[0] - outs[2]).abs().max().item()
    assert err <= bound, (err, bound)


@pytest.mark.parametrize("tokens,n_trees,T,K,splits,s,hidden,sde", [
    (1, 5, 3, 4, (0, 1), 2.0, 256, None),              # one token a node: up to 80 nodes in a tile, shared noise
    (48, 3, 4, 3, (0, 2), math.inf, 384, None),        # nodes that straddle tiles, clusters of three
    (130, 1, 4, 2, (1,), math.inf, 1024, (0, 1, 1, 0)),    # a tile of two tokens; ODE steps first and last
    (256, 2, 3, 1, (), math.inf, 1408, None),          # eleven chunks: not cut
    (4736, 2, 3, 2, (1,), math.inf, 256, None),        # 74 tiles in clusters of two, then 148: the step has its own launch
    (4737, 2, 2, 2, (0,), 1.0, 256, None),             # 75 tiles: not cut
])
def test_rollout_that_takes_the_step_along_is_the_step_by_step_rollout(B, tokens, n_trees, T, K, splits, s, hidden, sde):
    """Small frontiers: the velocity launch also makes the children.  Same noise, same float32 expressions, integer sums of
    squares: latents, velocity, log-probs and table are bit-equal to velocity and step in launches of their own."""
    from paper_2509_06040_b200.session import TreeSession
    w = Workload(name="along", n_trees=n_trees, tokens=tokens, channels=64, T=T, K=K, splits=splits, sigma=0.3,
                 velocity="mlp", reward="mixture", hidden=hidden, branch_corr_s=s)
    inp = make_inputs(w)
    flags = [1 if i in splits else 0 for i in range(T)]
    runs = []
    for along in (False, True, True):
        r = TreeSession(w, nodes_cap=w.nodes + 2)
        r.upload_inputs(inp)
        r.logp.fill_(7.0)
        r.init()
        if sde:
            B.tree_set_sde_steps(r.tree, list(sde))
        if along:
            B.tree_rollout(r.tree, flags, r.packed, hidden, r.v)
        else:
            for i in range(T):
                B.velocity_mlp(r.tree, r.packed, hidden, r.v)
                B.tree_step(r.tree, flags[i], r.v)
        B.tree_sync_status(r.tree)
        runs.append(r)
    n = n_trees * w.widths()[T - 1] * w.D
    for r in runs[1:]:
        assert torch.equal(r.latents[:, :w.nodes], runs[0].latents[:, :w.nodes])
        assert torch.equal(r.logp, runs[0].logp)
        assert torch.equal(r.node_table.view(4, n_trees, -1)[:, :, :w.nodes], runs[0].node_table.view(4, n_trees, -1)[:, :, :w.nodes])
        assert torch.equal(r.v.view(-1)[:n], runs[0].v.view(-1)[:n])


@pytest.mark.parametrize("tokens,n_trees,T,K,splits,hidden,sde", [
    (128, 300, 2, 1, (), 128, None),                   # a node is a tile; a third tile for four CTAs only
    (127, 400, 2, 1, (), 128, None),                   # less than a tile: the step has its own launch
    (1011, 38, 3, 2, (2,), 256, None),                 # 301 tiles, nodes end inside them, a last tile of 18 rows; then a fork, on its own
    (37889, 1, 4, 1, (), 128, (1, 0, 1, 0)),           # 297 tiles, one row in the last; ODE steps, the last one too
    (199, 1900, 2, 2, (0,), 128, None),                # 2 954 tiles: two children each, then 5 908
    (4096, 20, 3, 1, (), 1408, None),                  # eleven chunks, 640 tiles
    (5777, 2, 3, 2, (1,), 640, None),                  # 91 tiles, at most one to a CTA; a fork, on its own; 181 tiles
    (9600, 1, 3, 1, (), 512, (0, 1, 0)),               # four chunks; ODE steps first and last
    (9601, 1, 2, 1, (), 384, None),                    # three chunks: on its own
])
def test_children_of_whole_tiles_are_the_step_by_step_rollouts(B, tokens, n_trees, T, K, splits, hidden, sde):
    """Large frontiers: warps of the velocity launch make the children tile by tile.  The same bits as velocity and step in
    launches of their own, the velocities of the last step included."""
    test_rollout_that_takes_the_step_along_is_the_step_by_step_rollout(B, tokens, n_trees, T, K, splits, math.inf, hidden, sde)


@pytest.mark.parametrize("w1_std", [0.003, 0.02, 0.06, 0.12, 0.5])
def test_mlp_stage_against_64_bits(B, w1_std):
    """Against the unrounded GELU MLP of the bf16 latents in 64 bits.  Only the even half of an activation is rounded to bf16
    (2^-9 relative at most, as is its argument, which counts twice; 3.1e-4 the polynomial, 5e-4 the tanh form), and the roundings
    of the hidden units add up like independent ones: rms error <= sqrt(sum_j W2_j^2 e_j^2) with e_j the largest of each."""
    from paper_2509_06040_b200.session import TreeSession
    from workloads import Inputs, _to_bf16_values
    w = Workload(name="mlp_64", n_trees=1, tokens=600, channels=64, T=1, K=1, splits=(), sigma=0.3,
                 velocity="mlp", reward="mixture", hidden=1024)
    g = np.random.default_rng([5, int(w1_std * 1000)])
    W1 = _to_bf16_values(w1_std * g.standard_normal((64, 1024), dtype=np.float32))
    W2 = _to_bf16_values(0.02 * g.standard_normal((1024, 64), dtype=np.float32))
    s = TreeSession(w)
    s.upload_inputs(Inputs(W1=W1, W2=W2))
    s.init()
    B.velocity_mlp(s.tree, s.packed, w.hidden, s.v)
    B.tree_sync_status(s.tree)
    z = s.latents[0, 0].view(600, 64).to(torch.bfloat16).double()
    x = z @ torch.from_numpy(W1).cuda().double()
    W2d = torch.from_numpy(W2).cuda().double()
    ref = torch.nn.functional.gelu(x) @ W2d
    d = s.v.view(-1)[:ref.numel()].view_as(ref).double() - ref
    E = (x * torch.special.erf(x / 2 ** 0.5) / 2).abs()
    e = 2.0 ** -9 * 3 * E + 5e-4 * x.abs().clamp(max=1.0)
    bound = ((e ** 2) @ (W2d ** 2)).mean().sqrt().item() + 2.0 ** -16 * ref.pow(2).mean().sqrt().item()
    err = d.pow(2).mean().sqrt().item()
    print(f"w1_std {w1_std}: rms error {err / ref.pow(2).mean().sqrt().item():.2e} of rms(v), bound {bound:.2e}, is {err:.2e}")
    assert err <= bound


def test_replayed_rollout_gives_the_same_log_probs_every_time(B):
    """A rollout captured into a CUDA graph without the root kernel in front of it: every replay writes what the call writes
    (two tiles a level in clusters of eight, so the step goes along and its sums of squares are added with atomics)."""
    from paper_2509_06040_b200.session import TreeSession
    w = Workload(name="replay", n_trees=1, tokens=200, channels=64, T=4, K=2, splits=(0, 2), sigma=0.3,
                 velocity="mlp", reward="mixture", hidden=1024)
    inp = make_inputs(w)
    eager, s = TreeSession(w), TreeSession(w)
    for r in (eager, s):
        r.upload_inputs(inp)
        r.init()
    B.tree_rollout(eager.tree, eager._split_flags, eager.packed, w.hidden, eager.v)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.tree_rollout(s.tree, s._split_flags, s.packed, w.hidden, s.v)
    for _ in range(3):
        s.logp[:, 1:].fill_(7.0)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(s.logp, eager.logp) and torch.equal(s.latents, eager.latents)
    B.tree_sync_status(s.tree)


@pytest.mark.parametrize("tokens,channels,n_trees,T,K,splits,velocity,hidden,reward", [
    (16, 4, 1, 4, 2, (0, 2), "linear", 0, "neg_mse_target"),            # one-launch rollout and rewards
    (513, 4, 2, 8, 2, (0, 1, 2, 3, 4, 5, 6), "linear", 0, "mixture"),   # seven splits: step by step
    (300, 64, 2, 3, 2, (0,), "mlp", 1024, "normal_plus_cos"),           # the step goes along
    (45 * 128, 64, 1, 2, 1, (), "mlp", 1152, "mixture"),                # nine chunks: 45 tiles fit as clusters of three,
    (46 * 128, 64, 1, 2, 1, (), "mlp", 1152, "mixture"),                # 46 and 49 do not
    (49 * 128, 64, 1, 2, 1, (), "mlp", 1152, "neg_mse_target"),
])
def test_launches_of_a_pass_are_counted(B, tokens, channels, n_trees, T, K, splits, velocity, hidden, reward):
    """The session's count of a pass against the kernel nodes of the same pass captured into a graph."""
    from cuda.bindings import runtime
    from paper_2509_06040_b200.session import TreeSession
    w = Workload(name="count", n_trees=n_trees, tokens=tokens, channels=channels, T=T, K=K, splits=splits, sigma=0.3,
                 velocity=velocity, reward=reward, hidden=hidden or 3072)
    s = TreeSession(w)
    s.upload_inputs(make_inputs(w))
    s.run_all()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        s.run_all()
    raw = runtime.cudaGraph_t(graph.raw_cuda_graph())
    _, _, n = runtime.cudaGraphGetNodes(raw)
    _, nodes, n = runtime.cudaGraphGetNodes(raw, n)
    kernels = sum(1 for q in nodes if runtime.cudaGraphNodeGetType(q)[1] == runtime.cudaGraphNodeType.cudaGraphNodeTypeKernel)
    assert s.kernel_launches_per_pass() == kernels > 0
