"""Parity of the CUDA path (through the C ABI) against the CPU oracle, on the same seeded inputs.

Tolerances (stated by the target): Philox integers, node table and masks bit-exact; latents and
log-probs max abs error <= 1e-5; advantages <= 1e-4 relative (|d| <= 1e-4 * max(1, |A|)).
Reductions are tested teacher-forced as well: the oracle's float32 log-probs / rewards / fused
values are written into the device buffers, so the decision inputs are identical on both sides.
"""
import math

import numpy as np
import pytest
import torch

from oracle import credit, philox, rewards, sde
from oracle import tree as otree
from workloads import CONFIGS, Workload, make_inputs

pytestmark = pytest.mark.gpu

LATENT_TOL = 1e-5
LOGP_TOL = 1e-5
ADV_RTOL = 1e-4


@pytest.fixture(scope="module")
def B():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2509_06040_b200 import binding
    assert torch.cuda.is_available()
    return binding


def _session(w, **kw):
    from paper_2509_06040_b200.session import TreeSession
    return TreeSession(w, **kw)


def f32(x):
    return float(np.float32(x))


def oracle_rollout(w, inp, n_trees, tree_id_base=0, nodes_cap=None, velocity=None):
    """Oracle latents [n_trees][nodes][D], logp [n_trees][nodes] for the linear-velocity workloads
    (or any per-tree velocity callback factory `velocity(t)`)."""
    topo = otree.build_topology(w.T, w.K, w.splits)
    grid = w.t_grid().astype(np.float64)
    lats, logps = [], []
    for t in range(n_trees):
        if velocity is None:
            mu = inp.mu[t].astype(np.float64)
            vel = lambda z, i, p, mu=mu: sde.linear_velocity(z.astype(np.float64), float(grid[i]), mu, f32(w.s0))
        else:
            vel = velocity(t)
        lat, lp = sde.rollout(topo, w.D, grid, f32(w.sigma), w.branch_corr_s, w.seed, vel,
                              tree_id=tree_id_base + t, nodes_cap=nodes_cap or topo.nodes)
        lats.append(lat)
        logps.append(lp)
    return topo, np.stack(lats), np.stack(logps)


def assert_table(s, topo, n_trees):
    tab = s.node_table.cpu().numpy().reshape(4, n_trees, s.nodes_cap)
    for t in range(n_trees):
        assert np.array_equal(tab[0, t, :topo.nodes], topo.parent)
        assert np.array_equal(tab[1, t, :topo.nodes], topo.depth)
        assert np.array_equal(tab[2, t, :topo.nodes], topo.split_step)
        assert np.array_equal(tab[3, t, :topo.nodes], topo.branch_id)


def adv_close(got, ref):
    return np.all(np.abs(got - ref) <= ADV_RTOL * np.maximum(1.0, np.abs(ref)))


# ---------------------------------------------------------------------------------------------- noise
def test_philox_integer_stream_bit_exact(B):
    for seed, node, step, tag, nblk in ((0, 0, 0, 0, 64), (1223627, 154, 15, 2, 32400), ((7 << 32) | 9, 2 ** 32 - 1, 19, 1, 1000)):
        out = torch.empty((nblk, 4), dtype=torch.int32, device="cuda")
        B.philox_words_fill(seed, node, step, tag, out, nblk)
        got = out.cpu().numpy().view(np.uint32)
        assert np.array_equal(got, philox.noise_words(seed, node, step, tag, 4 * nblk))


def test_normals_match_float64_transform(B):
    n = 1 << 22
    out = torch.empty(n, dtype=torch.float32, device="cuda")
    B.philox_normal_fill(42, 77, 3, 2, out, n)
    got = out.cpu().numpy().astype(np.float64)
    ref = philox.node_noise(42, 77, 3, 2, n)
    err = np.abs(got - ref)
    # g <= 0.3 in every workload, so 2e-5 on xi is < 1e-5 on a latent; the observed error is far smaller
    assert err.max() < 2e-5, err.max()
    # the rare words whose uniform sits next to 1 (tiny radius) and next to 0 (largest radius) are present and accurate
    w = philox.noise_words(42, 77, 3, 2, n)
    ua = philox.uniform_open(w[:, 0])
    near_one = np.nonzero(1 - ua < 2.0 ** -9)[0]
    assert len(near_one) > 100 and err.reshape(-1, 4)[near_one].max() < 2e-5
    assert err.reshape(-1, 4)[np.argmin(ua)].max() < 2e-5


# ---------------------------------------------------------------------------------------------- toy config, end to end
def test_toy_config_end_to_end(B):
    w = CONFIGS["toy"]
    inp = make_inputs(w)
    s = _session(w)
    s.upload_inputs(inp)
    s.run_all()
    torch.cuda.synchronize()
    B.tree_sync_status(s.tree)
    topo, lat, logp = oracle_rollout(w, inp, 1)
    assert_table(s, topo, 1)
    assert np.abs(s.latents.cpu().numpy() - lat).max() <= LATENT_TOL
    assert np.abs(s.logp.cpu().numpy() - logp).max() <= LOGP_TOL
    r = np.array([rewards.neg_mse(lat[0][l], inp.mu[0]) for l in topo.leaf_ids()])
    assert np.abs(s.leaf_r.cpu().numpy()[0] - r).max() <= 1e-5
    rbar = credit.fuse_rewards(topo, r, logp[0], w.beta)
    adv = credit.depth_advantages(topo, rbar, f32(w.eps))
    assert np.abs(s.rbar.cpu().numpy()[0] - rbar).max() <= 1e-5
    assert adv_close(s.adv.cpu().numpy()[0], adv)
    assert np.array_equal(s.mask.cpu().numpy()[0], credit.gradient_mask(topo, rbar, w.width_mode, w.width_k))
    st = B.tree_stats(s.tree)
    assert (st["nodes"], st["node_steps"], st["model_evals"], st["frontier_width"]) == (13, 12, 9, 4)
    assert B.tree_levels(s.tree) == (topo.width, topo.offset[:-1])


# ---------------------------------------------------------------------------------------------- tiles, tails, K, s, batches
RAGGED = [
    # name, n_trees, tokens, channels, T, K, splits, sigma, s, tree_id_base, extra cap
    ("two_chunks_tail_k3_corr", 3, 2125, 4, 5, 3, (1, 3), 0.3, 2.0, 5, 7),
    ("k4_independent", 2, 1031, 4, 4, 4, (0, 3), 0.5, math.inf, 0, 0),
    ("k2_corr_s4_every_step", 1, 300, 4, 4, 2, (0, 1, 2, 3), 0.3, 4.0, 1000, 3),
    ("no_split_k1", 2, 9, 4, 6, 1, (), 0.7, math.inf, 0, 0),
    ("deterministic_sigma0", 1, 520, 4, 4, 2, (0, 2), 0.0, 1.0, 0, 0),
    ("exact_chunk_multiple", 1, 2048, 4, 3, 2, (1,), 0.3, math.inf, 2, 0),
]


def _grow(s, by_steps, seed=None):
    """A rollout of a closed-form session: tree_rollout, which takes one launch where it can, or tree_step depth by depth."""
    if not by_steps:
        return s.rollout(seed)
    s.init(seed)
    for i in range(s.w.T):
        s.step(i)


@pytest.mark.parametrize("by_steps", [False, True], ids=["one_call", "by_steps"])
@pytest.mark.parametrize("case", RAGGED, ids=[c[0] for c in RAGGED])
def test_rollout_parity_over_tiles_and_tails(B, case, by_steps):
    name, n_trees, tokens, channels, T, K, splits, sigma, s_corr, base, extra = case
    w = Workload(name=name, n_trees=n_trees, tokens=tokens, channels=channels, T=T, K=K, splits=splits, sigma=sigma,
                 velocity="linear", reward="neg_mse_mu", branch_corr_s=s_corr, seed=991 + T)
    inp = make_inputs(w, tree_base=base)
    cap = w.nodes + extra
    s = _session(w, tree_id_base=base, nodes_cap=cap)
    s.upload_inputs(inp)
    s.latents.fill_(float("nan"))
    _grow(s, by_steps)
    s.rewards()
    torch.cuda.synchronize()
    topo, lat, logp = oracle_rollout(w, inp, n_trees, tree_id_base=base, nodes_cap=cap)
    assert_table(s, topo, n_trees)
    got = s.latents.cpu().numpy()[:, :topo.nodes]
    assert np.abs(got - lat).max() <= LATENT_TOL
    assert np.abs(s.logp.cpu().numpy()[:, :topo.nodes] - logp).max() <= LOGP_TOL
    if extra:
        assert np.all(np.isnan(s.latents.cpu().numpy()[:, topo.nodes:]))      # rows beyond the tree are never written
    for t in range(n_trees):
        r = np.array([rewards.neg_mse(lat[t][l], inp.mu[t]) for l in topo.leaf_ids()])
        assert np.abs(s.leaf_r.cpu().numpy()[t] - r).max() <= 1e-5 * max(1.0, np.abs(r).max())
    # running the same handle again with the same seed reproduces every bit (fixed reduction order)
    first_lat, first_logp = s.latents.clone(), s.logp.clone()
    _grow(s, by_steps)
    torch.cuda.synchronize()
    assert torch.equal(first_logp[:, :topo.nodes], s.logp[:, :topo.nodes])
    assert torch.equal(first_lat[:, :topo.nodes], s.latents[:, :topo.nodes])
    # and another seed gives another tree
    _grow(s, by_steps, seed=12345)
    torch.cuda.synchronize()
    if sigma > 0:
        assert not torch.equal(first_lat[:, :topo.nodes], s.latents[:, :topo.nodes])


def test_sharded_batch_draws_the_same_noise(B):
    """Trees are independent: a shard with tree_id_base = t reproduces tree t of the whole batch."""
    w = Workload(name="shard", n_trees=4, tokens=64, channels=4, T=3, K=2, splits=(0, 2), sigma=0.3,
                 velocity="linear", reward="neg_mse_mu")
    whole = _session(w)
    whole.upload_inputs(make_inputs(w))
    whole.rollout()
    part = _session(w.scaled(n_trees=2), tree_id_base=2)
    part.upload_inputs(make_inputs(w.scaled(n_trees=2), tree_base=2))
    part.rollout()
    torch.cuda.synchronize()
    assert torch.equal(whole.latents[2:], part.latents)
    assert torch.equal(whole.logp[2:], part.logp)


def test_one_call_rollout_is_the_step_by_step_rollout(B):
    """bgrpo_tree_rollout makes what T x [velocity, tree_step] makes (Algorithm 1, "Build rollout tree"), a fresh closed-form
    tree in one launch: every output is identical bit for bit, for the closed-form and the MLP velocity, and it continues a
    tree that has already taken some steps."""
    for velocity, channels, hidden in (("linear", 4, 0), ("mlp", 64, 256)):
        w = Workload(name="one_call", n_trees=2, tokens=150, channels=channels, T=5, K=3, splits=(0, 3), sigma=0.3,
                     velocity=velocity, reward="mixture", hidden=hidden or 3072, branch_corr_s=2.0)
        inp = make_inputs(w)
        a, b, c = _session(w), _session(w), _session(w)
        for s in (a, b, c):
            s.upload_inputs(inp)
            s.init()
        flags = [1 if i in w.splits else 0 for i in range(w.T)]
        for i in range(w.T):                                   # a: one call per step
            a.step(i)
        if velocity == "mlp":                                  # b: one call for the tree; c: two steps, then the rest
            B.tree_rollout(b.tree, flags, b.packed, w.hidden, b.v)
            c.step(0); c.step(1)
            B.tree_rollout(c.tree, flags, c.packed, w.hidden, c.v)
        else:
            B.tree_rollout(b.tree, flags)
            c.step(0); c.step(1)
            B.tree_rollout(c.tree, flags)
        torch.cuda.synchronize()
        for s in (a, b, c):
            B.tree_sync_status(s.tree)
        for other in (b, c):
            assert B.tree_stats(other.tree) == B.tree_stats(a.tree)
            assert torch.equal(a.latents, other.latents) and torch.equal(a.logp[:, :w.nodes], other.logp[:, :w.nodes])
            assert torch.equal(a.node_table, other.node_table)
        with pytest.raises(B.BgrpoError) as e:                 # the tree is complete: nothing left to do is fine, a step is not
            B.tree_step(b.tree, 0, b.v if velocity == "mlp" else None)
        assert e.value.status == B.ERR_STATE
        B.tree_rollout(b.tree, flags, b.packed if velocity == "mlp" else None, w.hidden if velocity == "mlp" else 0, b.v)
    wl = Workload(name="one_call_err", n_trees=1, tokens=16, channels=4, T=2, K=2, splits=(0,), sigma=0.3, velocity="linear",
                  reward="neg_mse_mu")
    s = _session(wl)
    s.init()                                                    # no velocity bound, no weights given
    with pytest.raises(B.BgrpoError) as e:
        B.tree_rollout(s.tree, [1, 0])
    assert e.value.status == B.ERR_STATE


def test_export_import_continues_bit_identically(B):
    """A tree is saved after two steps (its host record plus copies of its device buffers, scratch left behind), restored
    into a new handle over the copies, and continued: every output equals the uninterrupted tree's bit for bit - for the
    closed-form velocity with the hybrid ODE-SDE schedule and for the MLP velocity."""
    for velocity, channels in (("linear", 4), ("mlp", 64)):
        w = Workload(name="resume", n_trees=2, tokens=150, channels=channels, T=5, K=2, splits=(0, 3), sigma=0.3,
                     velocity=velocity, reward="neg_mse_target", hidden=256, branch_corr_s=2.0, width_mode=B.WIDTH_PER_SPLIT_TOPK, width_k=1)
        inp = make_inputs(w)
        sde = [1, 0, 1, 1, 1]
        whole, first = _session(w, nodes_cap=w.nodes + 2), _session(w, nodes_cap=w.nodes + 2)
        for s in (whole, first):
            s.upload_inputs(inp)
            s.init()
            B.tree_set_sde_steps(s.tree, sde)
        for i in range(w.T):
            whole.step(i)
        first.step(0)
        first.step(1)
        blob = B.tree_export(first.tree)
        assert len(blob) == B.lib.bgrpo_tree_export_bytes()
        torch.cuda.synchronize()
        # the restored tree lives in copies of the buffers; its scratch is a fresh allocation
        second = _session(w, nodes_cap=w.nodes + 2)
        second.upload_inputs(inp)
        for name in ("latents", "node_table", "logp"):
            getattr(second, name).copy_(getattr(first, name))
        second.scratch.fill_(0xAB)
        second.tree = B.tree_import(blob, second.latents, second.node_table, second.logp, second.rbar, second.adv, second.mask, second.scratch)
        if velocity == "linear":
            B.velocity_linear_bind(second.tree, second.mu, f32(w.s0))
        assert B.tree_stats(second.tree) == B.tree_stats(first.tree)
        for i in range(2, w.T):
            second.step(i)
        for s in (whole, second):
            s.rewards(); s.fuse_advantage(); s.prune()
        torch.cuda.synchronize()
        B.tree_sync_status(second.tree)
        n = w.nodes
        assert torch.equal(whole.latents[:, :n], second.latents[:, :n])
        assert torch.equal(whole.logp[:, :n], second.logp[:, :n])
        cap = whole.nodes_cap
        assert torch.equal(whole.node_table.view(4, w.n_trees, cap)[:, :, :n], second.node_table.view(4, w.n_trees, cap)[:, :, :n])
        assert torch.equal(whole.leaf_r, second.leaf_r) and torch.equal(whole.adv[:, :n], second.adv[:, :n])
        assert torch.equal(whole.mask[:, :n], second.mask[:, :n])
    # a foreign record is refused
    with pytest.raises(B.BgrpoError) as e:
        B.tree_import(b"\0" * len(blob), second.latents, second.node_table, second.logp, second.rbar, second.adv, second.mask, second.scratch)
    assert e.value.status == B.ERR_INVALID_ARG


# ---------------------------------------------------------------------------------------------- given velocity (MLP stand-in path)
def test_step_with_supplied_velocity_and_logprob_recompute(B):
    """tree_step with a velocity buffer (the MLP configurations' path), teacher-forced: the oracle's MLP
    produces v for every frontier, both sides consume the same float32 v."""
    from oracle import mlp
    w = Workload(name="given_v", n_trees=2, tokens=40, channels=64, T=3, K=2, splits=(0, 2), sigma=0.3,
                 velocity="mlp", reward="mixture", hidden=128)
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

    lat, logp = [], []
    for t in range(w.n_trees):
        a, b = sde.rollout(topo, w.D, grid, f32(w.sigma), w.branch_corr_s, w.seed, vel_factory(t), tree_id=t, nodes_cap=topo.nodes)
        lat.append(a)
        logp.append(b)
    lat, logp = np.stack(lat), np.stack(logp)

    from paper_2509_06040_b200.session import TreeSession
    s = TreeSession(w)
    s.init()
    v_bufs = []
    for i in range(w.T):
        v = np.stack([np.stack([v_store[(t, i, p)] for p in topo.level(i)]) for t in range(w.n_trees)])
        v_dev = torch.from_numpy(v).cuda()
        v_bufs.append(v_dev)
        B.tree_step(s.tree, 1 if i in w.splits else 0, v_dev)
    torch.cuda.synchronize()
    assert np.abs(s.latents.cpu().numpy() - lat).max() <= LATENT_TOL
    assert np.abs(s.logp.cpu().numpy() - logp).max() <= LOGP_TOL
    # recompute under the same velocity: rho = 1
    out = torch.zeros_like(s.logp)
    for i in range(w.T):
        B.tree_logprob(s.tree, i, v_bufs[i], out)
    torch.cuda.synchronize()
    assert (out - s.logp).abs()[:, 1:].max().item() <= LOGP_TOL
    # under another velocity (a perturbed one): matches the oracle's edge log-prob of the stored latents
    i = 1
    v_new = v_bufs[i] + 0.05
    out2 = torch.full_like(s.logp, 7.0)
    B.tree_logprob(s.tree, i, v_new, out2)
    torch.cuda.synchronize()
    got = out2.cpu().numpy()
    v_new_h = v_new.cpu().numpy()
    for t in range(w.n_trees):
        for j, p in enumerate(topo.level(i)):
            for c in topo.children(p):
                ref = sde.edge_logp(lat[t][p], lat[t][c], v_new_h[t, j], grid[i], grid[i] - grid[i + 1], f32(w.sigma))
                assert abs(got[t, c] - ref) <= LOGP_TOL
        untouched = [n for n in range(topo.nodes) if topo.depth[n] != i + 1]
        assert np.all(got[t, untouched] == 7.0)


def test_logprob_all_edges_linear_velocity(B):
    w = Workload(name="lp_all", n_trees=2, tokens=700, channels=4, T=4, K=2, splits=(0, 2), sigma=0.3,
                 velocity="linear", reward="neg_mse_mu")
    inp = make_inputs(w)
    s = _session(w)
    s.upload_inputs(inp)
    s.rollout()
    out = torch.zeros_like(s.logp)
    B.tree_logprob(s.tree, -1, None, out)
    torch.cuda.synchronize()
    assert (out - s.logp)[:, 1:].abs().max().item() <= LOGP_TOL
    topo, lat, logp = oracle_rollout(w, inp, 2)
    assert np.abs(out.cpu().numpy()[:, 1:] - logp[:, 1:]).max() <= LOGP_TOL
    # a different policy (another target mean) against the oracle
    mu2 = torch.from_numpy(inp.mu + 0.1).cuda()
    B.velocity_linear_bind(s.tree, mu2, 0.5)
    B.tree_logprob(s.tree, -1, None, out)
    torch.cuda.synchronize()
    grid = w.t_grid().astype(np.float64)
    got = out.cpu().numpy()
    worst = 0.0
    for t in range(2):
        mu_h = (inp.mu[t] + np.float32(0.1)).astype(np.float64)
        for c in range(1, topo.nodes):
            p, i = int(topo.parent[c]), int(topo.depth[c]) - 1
            v = sde.linear_velocity(lat[t][p].astype(np.float64), grid[i], mu_h, 0.5)
            ref = sde.edge_logp(lat[t][p], lat[t][c], v, grid[i], grid[i] - grid[i + 1], f32(w.sigma))
            worst = max(worst, abs(got[t, c] - ref))
    print("worst |logp - oracle| under the perturbed policy:", worst)
    assert worst <= LOGP_TOL, worst


# ---------------------------------------------------------------------------------------------- rewards
def test_leaf_rewards(B):
    w = Workload(name="rw", n_trees=3, tokens=1500, channels=4, T=2, K=3, splits=(0, 1), sigma=0.3,
                 velocity="linear", reward="normal_plus_cos")
    inp = make_inputs(w)
    s = _session(w)
    s.upload_inputs(inp)
    s.rollout()
    s.rewards()
    torch.cuda.synchronize()
    topo, lat, _ = oracle_rollout(w, inp, 3)
    got = s.leaf_r.cpu().numpy()
    for t in range(3):
        for q, l in enumerate(topo.leaf_ids()):
            ref = float(inp.reward_draws[t, q]) + 0.1 * rewards.cosine(lat[t][l], inp.target[t])
            assert abs(got[t, q] - ref) <= 1e-6 * max(1.0, abs(ref))
    B.leaf_reward_mse(s.tree, s.target, s.leaf_r)
    torch.cuda.synchronize()
    got = s.leaf_r.cpu().numpy()
    for t in range(3):
        for q, l in enumerate(topo.leaf_ids()):
            ref = rewards.neg_mse(lat[t][l], inp.target[t])
            assert abs(got[t, q] - ref) <= 1e-6 * max(1.0, abs(ref))


# ---------------------------------------------------------------------------------------------- reductions, teacher-forced
def _grown_session(B, T, K, splits, n_trees=2, D_tokens=16):
    w = Workload(name="red", n_trees=n_trees, tokens=D_tokens, channels=4, T=T, K=K, splits=splits, sigma=0.3,
                 velocity="linear", reward="neg_mse_mu")
    s = _session(w)
    s.upload_inputs(make_inputs(w))
    s.rollout()
    return w, s, otree.build_topology(T, K, splits)


@pytest.mark.parametrize("T,K,splits", [(16, 2, (0, 3, 6, 9)), (6, 3, (0, 2, 5)), (5, 4, (1, 2, 4)), (20, 2, (0, 2, 4, 6, 8, 10)), (3, 2, ())])
def test_fuse_and_advantage_against_enumeration(B, T, K, splits):
    w, s, topo = _grown_session(B, T, K, splits)
    rng = np.random.default_rng(T * 10 + K)
    r = rng.standard_normal((2, topo.leaves)).astype(np.float32)
    r[1] = 3.0 + 1e-3 * r[1]                       # a tree whose rewards differ in the 4th digit only
    lp = (-np.abs(rng.standard_normal((2, topo.nodes))) - 0.3).astype(np.float32)
    lp[:, 0] = 0
    s.logp.copy_(torch.from_numpy(lp))
    r_dev = torch.from_numpy(r).cuda()
    for beta, scale, eps, clip in ((0.0, 1.0, 1e-6, 0.0), (1.0, 1.0, 1e-6, 0.0), (0.5, 64.0, 1e-3, 0.0), (1.0, 1.0, 1e-6, 0.8), (1.0, 1e5, 1e-6, 0.0)):
        B.tree_fuse_advantage(s.tree, r_dev, beta, scale, eps, clip)
        torch.cuda.synchronize()
        for t in range(2):
            rbar = credit.fuse_rewards(topo, r[t], lp[t].astype(np.float64), beta, scale)
            adv = credit.depth_advantages(topo, rbar, f32(eps), clip)
            got_rbar = s.rbar.cpu().numpy()[t]
            assert np.abs(got_rbar - rbar).max() <= 1e-6 * max(1.0, np.abs(rbar).max())
            assert adv_close(s.adv.cpu().numpy()[t], adv), (beta, scale, t)
            assert s.adv.cpu().numpy()[t, 0] == 0.0
    B.tree_sync_status(s.tree)


@pytest.mark.parametrize("T,K,splits", [(8, 3, (0, 2, 3, 4, 6)), (7, 3, (0, 1, 2, 3, 4, 5)), (4, 3, (2,)), (6, 2, (0, 2, 5)), (5, 4, (1, 3))])
def test_equal_rewards_have_no_advantage(B, T, K, splits):
    """All leaves of a tree with the same reward: every fused value is that reward and every advantage exactly zero (a sum of
    up to 729 equal float32 is exact in float64, and so is its correctly rounded quotient)."""
    w, s, topo = _grown_session(B, T, K, splits)
    for pair in ((0.1, 0.7), (1.0 / 3.0, -2.6), (1234.567, 1e-3), (0.0, 1.0)):
        r = np.repeat(np.array(pair, dtype=np.float32)[:, None], topo.leaves, axis=1)
        B.tree_fuse_advantage(s.tree, torch.from_numpy(np.ascontiguousarray(r)).cuda(), 0.0, 1.0, 1e-12, 0.0)
        torch.cuda.synchronize()
        assert np.array_equal(s.rbar.cpu().numpy(), np.repeat(r[:, :1], topo.nodes, axis=1)), pair
        assert not s.adv.cpu().numpy().any(), pair
    inf = torch.full((2, topo.leaves), float("inf"), device="cuda")      # an infinite reward stays what it was
    B.tree_fuse_advantage(s.tree, inf, 0.0, 1.0, 1e-6, 0.0)
    torch.cuda.synchronize()
    assert bool(torch.isinf(s.rbar).all())
    with pytest.raises(B.BgrpoError):
        B.tree_sync_status(s.tree)


@pytest.mark.parametrize("T,K,splits", [(16, 2, (0, 3, 6, 9)), (6, 4, (0, 2, 5)), (5, 3, (1, 2, 4)), (20, 2, (0, 5, 10))])
def test_prune_masks_bit_exact(B, T, K, splits):
    w, s, topo = _grown_session(B, T, K, splits)
    rng = np.random.default_rng(T + K)
    rbar = rng.standard_normal((2, topo.nodes)).astype(np.float32)
    rbar[1] = np.round(rbar[1])                    # many exact ties
    s.rbar.copy_(torch.from_numpy(rbar))
    s.adv.copy_(torch.from_numpy(rng.standard_normal(rbar.shape).astype(np.float32)))   # nothing has written it yet: a NaN left in that memory is not equal to itself
    before_adv, before_lat = s.adv.clone(), s.latents.clone()
    pruned = sorted(rng.choice(T, size=min(4, T), replace=False).tolist())
    cases = [(B.WIDTH_NONE, 0, (), False), (B.WIDTH_PER_SPLIT_TOPK, 1, (), False), (B.WIDTH_PER_SPLIT_TOPK, 2, pruned, False),
             (B.WIDTH_LAST_SPLIT_TOPK, 1, (), True), (B.WIDTH_EXTREME_B, 1, (), False), (B.WIDTH_EXTREME_B, 3, pruned, True),
             (B.WIDTH_EXTREME_B, 10 ** 6, (), False), (B.WIDTH_PER_SPLIT_TOPK, K, pruned, False)]
    for mode, k, pr, ign in cases:
        s.mask.fill_(9)
        B.tree_prune(s.tree, mode, k, pr, ign)
        torch.cuda.synchronize()
        got = s.mask.cpu().numpy()
        for t in range(2):
            ref = credit.gradient_mask(topo, rbar[t], mode, k, pr, ign)
            assert np.array_equal(got[t], ref), (mode, k, pr, ign, t)
    # pruning writes the mask only
    assert torch.equal(s.rbar.cpu(), torch.from_numpy(rbar))
    assert torch.equal(before_adv, s.adv) and torch.equal(before_lat, s.latents)


# ---------------------------------------------------------------------------------------------- states and errors
def test_state_and_capacity_errors(B):
    w = Workload(name="err", n_trees=1, tokens=16, channels=4, T=3, K=2, splits=(0, 1, 2), sigma=0.3,
                 velocity="linear", reward="neg_mse_mu")
    inp = make_inputs(w)
    s = _session(w, nodes_cap=11)                  # the full tree would need 15 rows
    s.upload_inputs(inp)
    s.init()
    r = torch.zeros((1, 8), device="cuda")
    with pytest.raises(B.BgrpoError) as e:
        B.tree_fuse_advantage(s.tree, r)
    assert e.value.status == B.ERR_STATE
    with pytest.raises(B.BgrpoError) as e:
        B.tree_prune(s.tree, B.WIDTH_NONE, 0)
    assert e.value.status == B.ERR_STATE
    with pytest.raises(B.BgrpoError) as e:
        B.tree_logprob(s.tree, 0, None, s.logp)
    assert e.value.status == B.ERR_STATE
    B.tree_step(s.tree, 1)
    B.tree_step(s.tree, 1)
    with pytest.raises(B.BgrpoError) as e:
        B.tree_step(s.tree, 1)                     # 1 + 2 + 4 + 8 > 11
    assert e.value.status == B.ERR_CAPACITY
    B.tree_step(s.tree, 0)                         # the refused call left the tree usable: 7 + 4 rows fit
    torch.cuda.synchronize()
    assert B.tree_stats(s.tree)["nodes"] == 11


def test_step_past_depth_and_missing_velocity(B):
    w = Workload(name="err2", n_trees=1, tokens=16, channels=4, T=2, K=2, splits=(0,), sigma=0.3,
                 velocity="linear", reward="neg_mse_mu")
    s = _session(w)
    s.init()                                        # no velocity bound
    with pytest.raises(B.BgrpoError) as e:
        B.tree_step(s.tree, 1)
    assert e.value.status == B.ERR_STATE
    s.upload_inputs(make_inputs(w))
    B.velocity_linear_bind(s.tree, s.mu, 0.5)
    B.tree_step(s.tree, 1)
    B.tree_step(s.tree, 0)
    with pytest.raises(B.BgrpoError) as e:
        B.tree_step(s.tree, 0)
    assert e.value.status == B.ERR_STATE
    torch.cuda.synchronize()


def test_nonfinite_reward_sets_status(B):
    w, s, topo = _grown_session(B, 3, 2, (0, 1), n_trees=1)
    r = torch.tensor([[0.0, 1.0, float("nan"), 2.0]], device="cuda")
    B.tree_fuse_advantage(s.tree, r)
    with pytest.raises(B.BgrpoError) as e:
        B.tree_sync_status(s.tree)
    assert e.value.status == B.ERR_NONFINITE
    B.tree_sync_status(s.tree)                     # the word is cleared by the read


# ---------------------------------------------------------------------------------------------- hybrid ODE-SDE schedule, Eq. 5
def test_hybrid_ode_sde_rollout_and_mask(B):
    w = Workload(name="mix", n_trees=2, tokens=600, channels=4, T=8, K=2, splits=(0, 3), sigma=0.3,
                 velocity="linear", reward="neg_mse_mu", seed=77)
    inp = make_inputs(w)
    sde_steps = B.mix_sde_steps(w.T, w.splits, iteration=60, window=2, every=30, start=4)      # splits + {6, 7}
    assert sde_steps == credit.mix_sde_steps(w.T, w.splits, 60, 2, 30, 4) == [0, 3, 6, 7]
    s = _session(w)
    s.upload_inputs(inp)
    s.init()
    B.tree_set_sde_steps(s.tree, [1 if i in sde_steps else 0 for i in range(w.T)])
    for i in range(w.T):
        s.step(i)
    s.rewards()
    s.fuse_advantage()
    s.prune()
    torch.cuda.synchronize()
    topo = otree.build_topology(w.T, w.K, w.splits)
    grid = w.t_grid().astype(np.float64)
    for t in range(2):
        mu = inp.mu[t].astype(np.float64)
        lat, logp = sde.rollout(topo, w.D, grid, f32(w.sigma), math.inf, w.seed,
                                lambda z, i, p: sde.linear_velocity(z.astype(np.float64), float(grid[i]), mu, 0.5),
                                tree_id=t, nodes_cap=topo.nodes, sde_steps=sde_steps)
        assert np.abs(s.latents[t].cpu().numpy() - lat).max() <= LATENT_TOL
        assert np.abs(s.logp[t].cpu().numpy() - logp).max() <= LOGP_TOL
        rbar = s.rbar[t].cpu().numpy()
        assert np.array_equal(s.mask[t].cpu().numpy(), credit.gradient_mask(topo, rbar, w.width_mode, w.width_k, (), False, sde_steps))
    # a split on an ODE step is refused, and the default (all SDE) can be restored
    s.init()
    B.tree_set_sde_steps(s.tree, [0] * w.T)
    with pytest.raises(B.BgrpoError) as e:
        B.tree_step(s.tree, 1)
    assert e.value.status == B.ERR_INVALID_ARG
    B.tree_set_sde_steps(s.tree, None)
    B.tree_step(s.tree, 1)
    torch.cuda.synchronize()


def test_grpo_objective_matches_oracle(B):
    w, s, topo = _grown_session(B, 8, 2, (0, 2, 5))
    rng = np.random.default_rng(8)
    adv = rng.standard_normal((2, topo.nodes)).astype(np.float32)
    mask = (rng.random((2, topo.nodes)) < 0.6).astype(np.uint8)
    mask[1, :] = 0                                   # a tree with an empty edge set
    old = (-np.abs(rng.standard_normal((2, topo.nodes))) - 0.2).astype(np.float32)
    new = (old + 0.01 * rng.standard_normal((2, topo.nodes))).astype(np.float32)
    s.adv.copy_(torch.from_numpy(adv))
    s.mask.copy_(torch.from_numpy(mask))
    s.logp.copy_(torch.from_numpy(old))
    new_dev = torch.from_numpy(new).cuda()
    J = torch.full((2,), 9.0, device="cuda")
    terms = torch.full_like(s.logp, 9.0)
    for eps, scale, use_buf in ((1e-4, 1.0, True), (0.2, 64.0, False)):
        B.tree_grpo_objective(s.tree, new_dev, None if use_buf else s.logp, scale, eps, terms, J)
        torch.cuda.synchronize()
        for t in range(2):
            Jr, tr = credit.grpo_objective(topo, new[t], old[t], adv[t], mask[t], f32(eps), f32(scale))
            assert abs(J[t].item() - Jr) <= 1e-6 * max(1.0, abs(Jr))
            assert np.abs(terms[t].cpu().numpy() - tr).max() <= 1e-6 * max(1.0, np.abs(tr).max())
    assert J[1].item() == 0.0


# ---------------------------------------------------------------------------------------------- whole-tree rollout in one launch
@pytest.mark.parametrize("tokens,channels,n_trees,T,K,splits,s,sigma", [
    (16, 4, 1, 4, 2, (0, 2), math.inf, 0.3),            # toy shape
    (700, 12, 2, 6, 2, (0, 2, 3), math.inf, 0.3),       # several chunks and a ragged tail (D/4 = 2100), consecutive splits
    (33, 20, 3, 5, 3, (1, 3), 2.0, 0.5),                # K = 3 with shared noise (finite s)
    (64, 16, 1, 7, 4, (6,), 1.0, 0.3),                  # K = 4, split at the last step
    (40, 8, 2, 6, 2, (0, 1, 2, 3, 4, 5), math.inf, 0.3),  # six splits: the deepest walk the kernel supports
    (24, 4, 1, 5, 1, (), math.inf, 0.3),                # no split at all
])
def test_fused_rollout_matches_oracle_and_stepwise(B, tokens, channels, n_trees, T, K, splits, s, sigma):
    w = Workload(name="fused", n_trees=n_trees, tokens=tokens, channels=channels, T=T, K=K, splits=splits, sigma=sigma,
                 velocity="linear", reward="neg_mse_mu", branch_corr_s=s)
    inp = make_inputs(w)
    topo, lat, logp = oracle_rollout(w, inp, n_trees)
    fused = _session(w, fused_rollout=True)
    fused.upload_inputs(inp)
    fused.rollout()
    step = _session(w)
    step.upload_inputs(inp)
    _grow(step, by_steps=True)
    torch.cuda.synchronize()
    B.tree_sync_status(fused.tree)
    assert_table(fused, topo, n_trees)
    assert B.tree_stats(fused.tree) == B.tree_stats(step.tree)
    got = fused.latents.cpu().numpy()[:, :topo.nodes]
    assert np.abs(got - lat).max() <= LATENT_TOL
    assert np.abs(fused.logp.cpu().numpy()[:, :topo.nodes] - logp).max() <= LOGP_TOL
    # the same draws and the same float32 expressions as the level-by-level kernel: identical latents
    assert np.array_equal(got, step.latents.cpu().numpy()[:, :topo.nodes])
    assert np.array_equal(fused.node_table.cpu().numpy(), step.node_table.cpu().numpy())
    # the reductions run on a tree grown either way
    fused.rewards(); fused.fuse_advantage(); fused.prune()
    step.rewards(); step.fuse_advantage(); step.prune()
    torch.cuda.synchronize()
    assert np.array_equal(fused.mask.cpu().numpy(), step.mask.cpu().numpy())
    assert np.allclose(fused.adv.cpu().numpy(), step.adv.cpu().numpy(), rtol=1e-4, atol=1e-4)


def test_fused_rollout_hybrid_schedule_and_errors(B):
    """ODE steps of the hybrid schedule (sigma = 0: child = mean, log-prob 0) and the call's error paths."""
    w = Workload(name="fused_mix", n_trees=1, tokens=50, channels=8, T=6, K=2, splits=(1, 3), sigma=0.3,
                 velocity="linear", reward="neg_mse_mu")
    inp = make_inputs(w)
    flags = [1 if i in w.splits else 0 for i in range(w.T)]
    sde_flags = [0, 1, 0, 1, 1, 0]
    a = _session(w)
    a.upload_inputs(inp)
    a.init()
    B.tree_set_sde_steps(a.tree, sde_flags)
    B.tree_rollout_fused(a.tree, flags)
    b = _session(w)
    b.upload_inputs(inp)
    b.init()
    B.tree_set_sde_steps(b.tree, sde_flags)
    for i in range(w.T):
        B.tree_step(b.tree, flags[i])
    torch.cuda.synchronize()
    assert np.array_equal(a.latents.cpu().numpy(), b.latents.cpu().numpy())
    assert np.abs(a.logp.cpu().numpy() - b.logp.cpu().numpy()).max() <= LOGP_TOL
    assert np.all(a.logp.cpu().numpy()[0, 1:2] == 0.0)                 # step 0 is an ODE step
    with pytest.raises(B.BgrpoError) as e:                             # the tree is complete
        B.tree_rollout_fused(a.tree, flags)
    assert e.value.status == B.ERR_STATE
    c = _session(w)
    c.upload_inputs(inp)
    c.init()
    B.tree_set_sde_steps(c.tree, [0, 0, 1, 1, 1, 1])
    with pytest.raises(B.BgrpoError) as e:                             # split on an ODE step
        B.tree_rollout_fused(c.tree, flags)
    assert e.value.status == B.ERR_INVALID_ARG
    w7 = Workload(name="fused7", n_trees=1, tokens=8, channels=4, T=7, K=2, splits=tuple(range(7)), sigma=0.3,
                  velocity="linear", reward="neg_mse_mu")
    d = _session(w7)
    d.upload_inputs(make_inputs(w7))
    d.init()
    with pytest.raises(B.BgrpoError) as e:                             # seven split steps
        B.tree_rollout_fused(d.tree, [1] * 7)
    assert e.value.status == B.ERR_UNSUPPORTED
    wm = Workload(name="fused_mlp", n_trees=1, tokens=8, channels=64, T=2, K=2, splits=(0,), sigma=0.3,
                  velocity="mlp", reward="mixture", hidden=128)
    m = _session(wm)
    m.upload_inputs(make_inputs(wm))
    m.init()
    with pytest.raises(B.BgrpoError) as e:                             # no bound closed-form velocity
        B.tree_rollout_fused(m.tree, [1, 0])
    assert e.value.status == B.ERR_STATE


# ---------------------------------------------------------------------------------------------- path-weighted fusion at scale, ESS, large trees
@pytest.mark.parametrize("T,K,splits", [(6, 3, (0, 1, 3, 4)), (5, 4, (0, 1, 2, 4)), (20, 3, (0, 3, 6, 9))])
def test_path_weighted_fusion_and_ess_on_wide_trees(B, T, K, splits):
    """K = 3 / 4 trees with 81 / 256 leaves (the paper's scaling study), beta = 1 (the ablation's path-probability
    weighting) on joint log-densities (logp_scale = D): fused values, advantages and the effective sample size of the
    weights against the oracle's enumeration, teacher-forced with the same float32 log-probs and rewards."""
    w, s, topo = _grown_session(B, T, K, splits, n_trees=2, D_tokens=8)
    assert topo.leaves in (81, 256)
    rng = np.random.default_rng(K * 100 + T)
    r = rng.standard_normal((2, topo.leaves)).astype(np.float32)
    lp = (-0.9 + 0.15 * rng.standard_normal((2, topo.nodes))).astype(np.float32)      # per-element means: close together
    lp[:, 0] = 0
    s.logp.copy_(torch.from_numpy(lp))
    r_dev = torch.from_numpy(r).cuda()
    ess = torch.empty_like(s.logp)
    for beta, scale in ((1.0, float(w.D)), (0.0, 1.0), (2.5, 1.0)):
        B.tree_fuse_advantage(s.tree, r_dev, beta, scale, 1e-6, 0.0)
        B.tree_fusion_ess(s.tree, beta, scale, ess)
        torch.cuda.synchronize()
        for t in range(2):
            rbar = credit.fuse_rewards(topo, r[t], lp[t].astype(np.float64), beta, scale)
            adv = credit.depth_advantages(topo, rbar, 1e-6)
            ref_ess = credit.fusion_ess(topo, lp[t].astype(np.float64), beta, scale)
            assert np.abs(s.rbar.cpu().numpy()[t] - rbar).max() <= 1e-6 * max(1.0, np.abs(rbar).max())
            assert adv_close(s.adv.cpu().numpy()[t], adv), (beta, scale, t)
            got_ess = ess.cpu().numpy()[t, :topo.nodes]
            assert np.all(np.abs(got_ess - ref_ess) <= 1e-5 * ref_ess), (beta, scale, t)
            if beta == 0.0:
                assert got_ess[0] == topo.leaves
    B.tree_sync_status(s.tree)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_ess_has_no_value_above_an_edge_that_is_not_finite(B, bad):
    """A log-prob that is not finite leaves the effective sample size of every node above its edge without a value, wherever on
    a chain the edge lies, and all other nodes untouched.  Minus infinity below a fork is a weight of zero among others."""
    w, s, topo = _grown_session(B, 12, 2, (1, 6), n_trees=1)
    lp = np.full(topo.nodes, -0.9, dtype=np.float32)
    ess, ref = torch.empty_like(s.logp), torch.empty_like(s.logp)
    s.logp.copy_(torch.from_numpy(lp[None]))
    B.tree_fusion_ess(s.tree, 1.0, 1.0, ref)
    for n in [1] + [int(topo.level(d)[-1]) for d in (2, 4, 6, 7, 9, 12)]:      # edges into: the first chain, both forks' children, mid-chain, a leaf
        lp_n = lp.copy()
        lp_n[n] = bad
        s.logp.copy_(torch.from_numpy(lp_n[None]))
        B.tree_fusion_ess(s.tree, 1.0, 1.0, ess)
        torch.cuda.synchronize()
        above, q = set(), int(topo.parent[n])
        while q >= 0:
            above.add(q)
            q = int(topo.parent[q])
        no_weight = bad == float("-inf") and int(topo.depth[n]) - 1 in (1, 6)
        for q in range(topo.nodes):
            got = float(ess[0, q])
            if q in above:
                assert got < float(ref[0, q]) if no_weight else math.isnan(got), (n, q, got)
            else:
                assert got == float(ref[0, q]), (n, q, got)


def test_reductions_on_a_tree_larger_than_shared_memory(B):
    """K = 4 with seven splits: 21 845 nodes, more than one CTA's shared memory holds as doubles; the reduction kernels
    keep their per-node state in the caller's scratch instead.  Fusion, advantages, ESS and masks against the oracle."""
    T, K, splits = 7, 4, tuple(range(7))
    w = Workload(name="huge", n_trees=2, tokens=1, channels=4, T=T, K=K, splits=splits, sigma=0.3,
                 velocity="linear", reward="neg_mse_mu")
    s = _session(w)
    s.upload_inputs(make_inputs(w))
    s.rollout()
    topo = otree.build_topology(T, K, splits)
    assert topo.nodes == 21845 and topo.nodes * 16 > 200 * 1024
    rng = np.random.default_rng(77)
    r = rng.standard_normal((2, topo.leaves)).astype(np.float32)
    lp = (-1.0 + 0.4 * rng.standard_normal((2, topo.nodes))).astype(np.float32)
    lp[:, 0] = 0
    s.logp.copy_(torch.from_numpy(lp))
    r_dev = torch.from_numpy(r).cuda()
    ess = torch.empty_like(s.logp)
    beta = 1.0
    B.tree_fuse_advantage(s.tree, r_dev, beta, 1.0, 1e-6, 0.0)
    B.tree_fusion_ess(s.tree, beta, 1.0, ess)
    B.tree_prune(s.tree, B.WIDTH_PER_SPLIT_TOPK, 2, (1, 4), False)
    torch.cuda.synchronize()
    B.tree_sync_status(s.tree)
    t = 1
    rbar = credit.fuse_rewards(topo, r[t], lp[t].astype(np.float64), beta, 1.0)
    adv = credit.depth_advantages(topo, rbar, 1e-6)
    assert np.abs(s.rbar.cpu().numpy()[t] - rbar).max() <= 1e-6 * max(1.0, np.abs(rbar).max())
    assert adv_close(s.adv.cpu().numpy()[t], adv)
    ref_ess = credit.fusion_ess(topo, lp[t].astype(np.float64), beta, 1.0)
    assert np.all(np.abs(ess.cpu().numpy()[t] - ref_ess) <= 1e-5 * ref_ess)
    mask = credit.gradient_mask(topo, s.rbar.cpu().numpy()[t], B.WIDTH_PER_SPLIT_TOPK, 2, (1, 4), False)
    assert np.array_equal(s.mask.cpu().numpy()[t], mask)
    # Extreme-b on the 16 384 leaves of this tree (a CTA-wide selection of the b-th best and b-th worst leaf), with
    # exact ties: values rounded to one decimal, signed zeros included
    coarse = np.round(s.rbar.cpu().numpy(), 1).astype(np.float32)
    s.rbar.copy_(torch.from_numpy(coarse))
    for b, pruned, ign in ((1, (), False), (37, (2,), True), (5000, (), False), (10 ** 6, (0, 6), False)):
        s.mask.fill_(9)
        B.tree_prune(s.tree, B.WIDTH_EXTREME_B, b, pruned, ign)
        torch.cuda.synchronize()
        got = s.mask.cpu().numpy()
        for t in range(2):
            ref = credit.gradient_mask(topo, coarse[t], B.WIDTH_EXTREME_B, b, pruned, ign)
            assert np.array_equal(got[t], ref), (b, t)
            if not pruned and not ign:
                assert int(got[t][list(topo.leaf_ids())].sum()) == min(2 * b, topo.leaves)


def test_prune_has_no_node_limit(B):
    """A tree of 349 525 nodes (K = 4, nine splits): every pruning mode runs (the values stay in global memory, the
    Extreme-b flags are gathered in the mask itself) and matches the oracle."""
    T, K, splits = 9, 4, tuple(range(9))
    w = Workload(name="huge9", n_trees=1, tokens=1, channels=4, T=T, K=K, splits=splits, sigma=0.3,
                 velocity="linear", reward="neg_mse_mu")
    s = _session(w)
    s.upload_inputs(make_inputs(w))
    s.rollout()
    topo = otree.build_topology(T, K, splits)
    assert topo.nodes == 349525
    rng = np.random.default_rng(5)
    rbar = np.round(rng.standard_normal((1, topo.nodes)), 2).astype(np.float32)
    s.rbar.copy_(torch.from_numpy(rbar))
    for mode, k in ((B.WIDTH_EXTREME_B, 3), (B.WIDTH_LAST_SPLIT_TOPK, 1)):
        B.tree_prune(s.tree, mode, k, (4,), False)
        torch.cuda.synchronize()
        ref = credit.gradient_mask(topo, rbar[0], mode, k, (4,), False)
        assert np.array_equal(s.mask.cpu().numpy()[0], ref), mode


@pytest.mark.parametrize("T,K,splits", [(1, 2, ()), (1, 3, (0,)), (9, 2, tuple(range(9))), (12, 2, (0, 1, 2, 3, 4, 5, 6, 8, 9, 10)), (8, 1, (2, 5)),
                                        (7, 4, (0, 1, 3, 4, 5)), (9, 4, (0, 1, 4, 6)), (11, 3, (0, 2, 3, 5, 7)), (10, 2, tuple(range(8)))])
def test_reductions_where_their_branches_change(B, T, K, splits):
    """Trees at the edges of the reductions' branches: one run only, forks at every step, long chains, K = 1 "forks", and
    Extreme-b on 512 leaves (ranked by counting) and 1024 (radix selection), with exact ties; runs of 243, 256 and more chains
    (masks written node by node, chain by chain).  Masks are whole numbers;
    fused values, advantages and effective sample sizes within the bounds of the tests above."""
    w, s, topo = _grown_session(B, T, K, splits)
    rng = np.random.default_rng(100 * T + K)
    r = np.round(rng.standard_normal((2, topo.leaves)), 1).astype(np.float32)
    lp = (-0.9 + 0.3 * rng.standard_normal((2, topo.nodes))).astype(np.float32)
    lp[:, 0] = 0
    s.logp.copy_(torch.from_numpy(lp))
    ess = torch.empty_like(s.logp)
    for beta in (0.0, 1.0):
        B.tree_fuse_advantage(s.tree, torch.from_numpy(r).cuda(), beta, 1.0, 1e-6, 5.0)
        B.tree_fusion_ess(s.tree, beta, 1.0, ess)
        torch.cuda.synchronize()
        for t in range(2):
            rbar = credit.fuse_rewards(topo, r[t], lp[t].astype(np.float64), beta, 1.0)
            ref_ess = credit.fusion_ess(topo, lp[t].astype(np.float64), beta, 1.0)
            assert np.abs(s.rbar.cpu().numpy()[t] - rbar).max() <= 1e-6 * max(1.0, np.abs(rbar).max())
            assert adv_close(s.adv.cpu().numpy()[t], credit.depth_advantages(topo, rbar, f32(1e-6), 5.0))
            assert np.all(np.abs(ess.cpu().numpy()[t, :topo.nodes] - ref_ess) <= 1e-5 * ref_ess)
    coarse = np.round(rng.standard_normal((2, topo.nodes)), 1).astype(np.float32)
    s.rbar.copy_(torch.from_numpy(coarse))
    for mode, k in ((B.WIDTH_EXTREME_B, 1), (B.WIDTH_EXTREME_B, 100), (B.WIDTH_PER_SPLIT_TOPK, 1), (B.WIDTH_LAST_SPLIT_TOPK, 2)):
        s.mask.fill_(9)
        B.tree_prune(s.tree, mode, k, (T - 1,), False)
        torch.cuda.synchronize()
        for t in range(2):
            assert np.array_equal(s.mask.cpu().numpy()[t], credit.gradient_mask(topo, coarse[t], mode, k, (T - 1,), False)), (mode, k, t)
    B.tree_sync_status(s.tree)


@pytest.mark.parametrize("tokens,channels,n_trees,T,K,splits,grown", [
    (1, 4, 1, 3, 2, (1,), 3),                 # one float4 a row
    (512, 4, 2, 5, 3, (0, 3), 5),             # exactly one chunk a row
    (513, 4, 1, 6, 4, (2,), 4),               # one float4 more; a partly grown tree that ends in a chain
    (1021, 16, 2, 4, 2, (0, 1, 2, 3), 4),     # ragged last chunk, no chains
    (300, 64, 3, 7, 2, (), 7),                # no fork at all
])
def test_logprob_families_at_their_edges(B, tokens, channels, n_trees, T, K, splits, grown):
    """Stored edges scored per step and all at once (families walked down the chains), closed form and supplied velocity,
    against the float64 formula on the stored latents; each call twice."""
    w = Workload(name="families", n_trees=n_trees, tokens=tokens, channels=channels, T=T, K=K, splits=splits, sigma=0.3,
                 velocity="linear", reward="neg_mse_mu")
    s = _session(w)
    s.upload_inputs(make_inputs(w))
    s.init()
    for i in range(grown):
        s.step(i)
    widths, offs = B.tree_levels(s.tree)
    g = torch.Generator(device="cuda").manual_seed(tokens)
    lat, mu, grid, sig, s0 = s.latents.double(), s.mu.double(), w.t_grid().astype(np.float64), f32(w.sigma), f32(w.s0)
    every = torch.full_like(s.logp, 7.0)
    B.tree_logprob(s.tree, -1, None, every)
    for i in range(grown):
        W, F = widths[i], widths[i + 1] // widths[i]
        t, h = grid[i], grid[i] - grid[i + 1]
        z = lat[:, offs[i]:offs[i] + W]
        child = lat[:, offs[i + 1]:offs[i + 1] + W * F].view(n_trees, W, F, w.D)
        k = (t - (1 - t) * s0 * s0) / ((1 - t) ** 2 * s0 * s0 + t * t)
        v_lin = -mu[:, None] + k * (z - (1 - t) * mu[:, None])
        v_given = torch.randn(n_trees, W, w.D, device="cuda", generator=g)
        for v, given in ((v_lin, None), (v_given.double(), v_given)):
            mean = z - h * v - sig * sig * h / (2 * t) * (z + (1 - t) * v)
            ref = -((child - mean[:, :, None]) ** 2).mean(-1) / (2 * sig * sig * h) - math.log(sig * math.sqrt(h)) - 0.5 * math.log(2 * math.pi)
            ref = ref.view(n_trees, W * F)
            bound = 1e-5 * ref.abs().clamp(min=1.0)
            got = torch.full_like(s.logp, 7.0)
            for _ in range(2):
                B.tree_logprob(s.tree, i, given, got)
            rows = slice(offs[i + 1], offs[i + 1] + W * F)
            assert bool(((got[:, rows].double() - ref).abs() <= bound).all()), i
            if given is None:
                assert bool(((every[:, rows].double() - ref).abs() <= bound).all()), i
            got[:, rows] = 7.0
            assert bool((got == 7.0).all())                 # only the addressed edges were written
    assert bool((every[:, 0] == 7.0).all())
    B.tree_sync_status(s.tree)


@pytest.mark.parametrize("tokens,channels,n_trees,T,K,splits,s", [
    (9, 4, 591, 2, 1, (), math.inf),              # step launches of 591, 592, 593 CTAs: the small ones and the large ones
    (9, 4, 592, 2, 1, (), math.inf),
    (9, 4, 593, 2, 1, (), math.inf),
    (513, 4, 295, 2, 1, (), math.inf),            # the same with a second chunk of one float4 (two-CTA rows in the whole-tree launch)
    (513, 4, 296, 2, 1, (), math.inf),
    (512, 4, 147, 3, 4, (0,), 2.0),               # a full chunk, four children, shared noise; 588 and 592 CTAs in the steps after the fork
    (512, 4, 148, 3, 4, (0,), 2.0),
    (1, 4, 3, 4, 3, (0, 2), 1.0),                 # one float4 a row; every fork dealt out to the grid
    (9, 4, 1, 20, 2, (0, 1, 2, 3, 4, 5), math.inf),   # 1023 nodes: the rows' sums stay in shared memory
    (9, 4, 1, 21, 2, (0, 1, 2, 3, 4, 5), math.inf),   # 1087 nodes: they do not
    (9, 4, 450, 6, 2, (0, 1, 2, 3, 4, 5), 2.0),   # two forks dealt out, four open ones with their shared noise in shared memory
    (9, 4, 444, 7, 2, (1, 2, 3, 4, 5, 6), 2.0),   # three trees an SM, no fork dealt out: six open forks
    (513, 4, 444, 7, 2, (1, 2, 3, 4, 5, 6), 2.0),     # the same with rows of two CTAs
    (128, 4, 3, 4, 3, (0, 2), 1.0),               # the whole-tree launch takes one float4 a thread, two, two, four
    (129, 4, 3, 4, 4, (0, 2), 2.0),
    (256, 4, 2, 5, 2, (0, 3), math.inf),
    (257, 4, 2, 5, 2, (0, 3), 2.0),
    (513, 4, 148, 3, 2, (), 2.0),                 # no fork: one float4 a thread, and four with one tree more
    (513, 4, 149, 3, 2, (), 2.0),
    (63 * 512, 4, 1, 3, 2, (1,), math.inf),       # sums of 504 and 520 numbers a row: the last launch takes a warp or a CTA per row
    (64 * 512 + 1, 4, 1, 3, 2, (1,), math.inf),
    (127 * 512, 4, 5, 3, 2, (1,), math.inf),      # 508 and 512 of the wide launches
    (128 * 512, 4, 5, 3, 2, (1,), 2.0),
])
def test_step_and_whole_tree_launches_agree_where_their_shapes_change(B, tokens, channels, n_trees, T, K, splits, s):
    """The two rollouts share the noise stream, the float32 expressions and the integer sums, and nothing of their launch
    shapes: latents, log-probs and tables are bit-equal.  (Both are compared with the oracle above.)"""
    w = Workload(name="shapes", n_trees=n_trees, tokens=tokens, channels=channels, T=T, K=K, splits=splits, sigma=0.3,
                 velocity="linear", reward="neg_mse_mu", branch_corr_s=s)
    inp = make_inputs(w)
    runs = []
    for fused in (False, True):
        r = _session(w, fused_rollout=fused)
        r.upload_inputs(inp)
        r.logp.fill_(7.0)
        if fused:
            r.rollout()
        else:
            r.init()
            for i in range(T):
                r.step(i)
        B.tree_sync_status(r.tree)
        runs.append(r)
    step, whole = runs
    assert torch.equal(step.latents, whole.latents)
    assert torch.equal(step.logp, whole.logp)
    assert torch.equal(step.node_table, whole.node_table)


@pytest.mark.parametrize("tokens,channels", [(1, 4), (4096, 4), (4097, 4), (8193, 4)])      # rows of one, one, two and three chunks
def test_leaf_rewards_where_a_row_outgrows_its_cta(B, tokens, channels):
    w = Workload(name="rw", n_trees=2, tokens=tokens, channels=channels, T=2, K=2, splits=(0,), sigma=0.3,
                 velocity="linear", reward="normal_plus_cos")
    inp = make_inputs(w)
    s = _session(w)
    s.upload_inputs(inp)
    s.rollout()
    leaf = s.latents[:, -w.leaves:].double()
    target = s.target.double().view(2, 1, w.D)
    cos = (leaf * target).sum(-1) / (leaf.norm(dim=-1) * target.norm(dim=-1))
    refs = (torch.from_numpy(inp.reward_draws).cuda().double() + 0.1 * cos, -((leaf - target) ** 2).mean(-1))
    for _ in range(2):
        s.rewards()
        got = [s.leaf_r.clone()]
        B.leaf_reward_mse(s.tree, s.target, s.leaf_r)
        got.append(s.leaf_r.clone())
        for g, ref in zip(got, refs):         # sums in float64, one rounding to float32
            assert bool(((g.double() - ref).abs() <= 1e-6 * ref.abs().clamp(min=1.0)).all())
