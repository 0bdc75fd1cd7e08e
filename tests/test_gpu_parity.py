"""GPU parity tests: the CUDA library (through its C ABI) against the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_2107_01460_b200 import binding, workloads as wl

from parity import GAE_TOL, check_against_oracle, run_gpu

pytestmark = pytest.mark.gpu

FP32 = binding.MAVA_PRECISION_FP32
BF16 = binding.MAVA_PRECISION_BF16


def _precision(w):
    return BF16 if w["precision"] == "bf16" else FP32


def _tc_available(w):
    import ctypes as C

    cfg = binding.make_config(w, precision=BF16)
    return bool(binding.lib().mava_params_count(C.byref(cfg))) and _try_create(cfg)


def _try_create(cfg):
    try:
        cfg2 = binding.mava_config_t.from_buffer_copy(cfg)
        cfg2.n_envs, cfg2.max_T = 4, 2
        binding.Rollout(cfg2).close()
        return True
    except binding.MavaError as e:
        if e.code == binding.MAVA_ERR_UNSUPPORTED:
            return False
        raise


# ---- whole small config, every environment checked -------------------------------------------

@pytest.mark.parametrize("bias_scale", [0.0, 0.5])
def test_cfg0_fp32_every_row(bias_scale):
    w = wl.workload(0)
    params = wl.make_params(w, bias_scale=bias_scale)
    ro, _ = run_gpu(w, FP32, w["T"], params=params)
    out = check_against_oracle(w, ro, params, w["T"], FP32, np.arange(w["n_envs"]))
    print(out)


def test_cfg0_longer_than_the_cap_crosses_resets():
    w = wl.workload(0)
    params = wl.make_params(w)
    T = 120
    ro, _ = run_gpu(w, FP32, T, params=params)
    assert int(ro.dones.sum()) >= 2 * w["n_envs"]
    check_against_oracle(w, ro, params, T, FP32, np.arange(w["n_envs"]))


# ---- reduced versions of the larger configs (several tiles and a ragged last tile) -----------

@pytest.mark.parametrize("idx,n_envs,T", [(1, 77, 60), (2, 101, 110), (3, 45, 105), (4, 37, 40)])
def test_reduced_configs_fp32(idx, n_envs, T):
    w = wl.workload(idx)
    params = wl.make_params(w, bias_scale=0.1)
    ro, _ = run_gpu(w, FP32, T, n_envs=n_envs, params=params)
    ids = wl.sample_env_ids(n_envs, 6, 6, 6, seed=idx)
    out = check_against_oracle(w, ro, params, T, FP32, ids)
    print(idx, out)


@pytest.mark.parametrize("idx,n_envs,T,mode", [(1, 333, 60, ""), (2, 300, 110, ""), (3, 200, 105, ""),
                                               (4, 150, 40, ""), (0, 16, 32, "tmem"), (1, 333, 60, "tmem"),
                                               (2, 300, 110, "tmem"), (1, 333, 60, "wide"), (2, 300, 110, "wide"),
                                               (1, 1500, 40, ""), (2, 1000, 40, ""), (1, 1500, 40, "wide"),
                                               # H = 256 with more tiles than one round holds and an odd count: a second
                                               # round in which one thread group of a CTA has no tile (on 148 SMs)
                                               (4, 4737, 12, ""), (3, 9473, 7, "")])
def test_reduced_configs_bf16(idx, n_envs, T, mode):
    """"wide" and "tmem" (two flags that ask for the same) force 128-row tiles where the batch is small enough for the few-rows
    form of the kernel (up to 16 rows per SM at 16 / 333 / 300 environments, up to 32 at 1500 / 1000)."""
    w = wl.workload(idx)
    if not _tc_available(w):
        pytest.skip("bf16 tensor-core path not compiled for this shape")
    params = wl.make_params(w, bias_scale=0.1)
    flags = binding.MAVA_FLAG_WRITE_LOGITS | {"": 0, "tmem": binding.MAVA_FLAG_HIDDEN_IN_TMEM,
                                              "wide": binding.MAVA_FLAG_WIDE_TILES}[mode]
    ro, _ = run_gpu(w, BF16, T, n_envs=n_envs, params=params, flags=flags)
    ids = wl.sample_env_ids(n_envs, 6, 6, 6, seed=idx)
    out = check_against_oracle(w, ro, params, T, BF16, ids)
    print(idx, out)


@pytest.mark.parametrize("idx,n_envs", [(1, 1024), (1, 2000), (2, 700), (2, 1400), (0, 16), (0, 1185), (0, 2368),
                                         ("wh0_tiny_8x8_2r2s_h64", 16), ("wh1_10x10_3r3s_h128", 741), ("wh2_10x10_3r3s_h128_collisions_end", 1480)])
def test_few_rows_form_equals_wide_tiles(idx, n_envs):
    """The few-rows form of the bf16 kernel (rows as the N operand of the MMA) forms the same products
    in the same order as the 128-row form: every output is bit-identical.  Workload 0: its 64 units padded to 128."""
    w = wl.workload(idx)
    T = 48
    params = wl.make_params(w, bias_scale=0.1)
    outs = []
    for extra in (0, binding.MAVA_FLAG_WIDE_TILES):
        ro, _ = run_gpu(w, BF16, T, n_envs=n_envs, params=params, flags=binding.MAVA_FLAG_WRITE_LOGITS | extra)
        outs.append({k: getattr(ro, k)[:T + (1 if k == "values" else 0)].cpu().numpy().copy()
                     for k in ("obs", "actions", "logp", "values", "rewards", "dones", "logits", "adv", "ret")})
    for k in outs[0]:
        assert np.array_equal(outs[0][k].view(np.uint8), outs[1][k].view(np.uint8)), k


@pytest.mark.parametrize("name,n_envs,grid,cap,T,wide", [
    # the smallest worlds that take their agents and foods, and the largest (a byte per coordinate: the window's
    # out-of-range rows and columns are found by byte arithmetic); episodes of one and of a few steps; odd batches, so that
    # a warp's or a tile's observation block is not a whole number of 16-byte pieces
    ("cfg1_8x8_2p2f_h128", 7, 3, 1, 5, False), ("cfg1_8x8_2p2f_h128", 301, 64, 3, 9, False),
    ("cfg1_8x8_2p2f_h128", 1333, 4, 2, 6, False), ("cfg1_8x8_2p2f_h128", 301, 3, 3, 9, True),
    ("cfg1_8x8_2p2f_h128", 2401, 64, 5, 12, False), ("cfg2_10x10_3p3f_h128", 149, 3, 2, 7, False),
    ("cfg2_10x10_3p3f_h128", 1511, 64, 4, 9, False), ("cfg0_tiny_8x8_2p2f_h64", 5, 3, 1, 3, False),
    ("cfg0_tiny_8x8_2p2f_h64", 333, 64, 7, 15, False), ("cfg3_15x15_4p5f_mappo_h256", 31, 3, 3, 7, False),
    ("cfg4_20x20_8p8f_h256", 37, 4, 2, 5, False), ("cfg4_20x20_8p8f_h256", 19, 64, 3, 7, False),
    # H = 256 around one full tile per SM (148 SMs): the largest batch for one thread group, the smallest for two
    ("cfg4_20x20_8p8f_h256", 2368, 20, 3, 5, False), ("cfg4_20x20_8p8f_h256", 2369, 20, 3, 5, False),
    ("rec1_8x8_2p2f_gru64", 37, 3, 2, 7, False), ("rec1_8x8_2p2f_gru64", 131, 64, 4, 9, False),
    ("wh1_10x10_3r3s_h128", 61, 4, 3, 9, False), ("wh1_10x10_3r3s_h128", 301, 64, 5, 11, False),
    ("wh2_10x10_3r3s_h128_collisions_end", 501, 5, 4, 13, False)])
def test_bf16_worlds_at_the_ends_of_their_range(name, n_envs, grid, cap, T, wide):
    w = dict(wl.workload(name), grid=grid, episode_cap=cap)
    params = wl.make_params(w, bias_scale=0.1)
    flags = binding.MAVA_FLAG_WRITE_LOGITS | (binding.MAVA_FLAG_WIDE_TILES if wide else 0)
    if w["net_kind"] == 2:  # the recurrent oracle has its own comparison: environment arrays only
        ro, _ = run_gpu(w, BF16, T, n_envs=n_envs, params=params, flags=flags)
        acts = ro.actions[:T].cpu().numpy()
        ref = oracle.rollout(oracle.make_config(w), w["seed"], None, T, np.arange(n_envs, dtype=np.int32),
                             forced_actions=acts, compute_mlp=False)
        assert np.array_equal(ref.obs.view(np.uint32), ro.obs[:T].cpu().numpy().view(np.uint32))
        assert np.array_equal(ref.rewards.view(np.uint32), ro.rewards[:T].cpu().numpy().view(np.uint32))
        assert np.array_equal(ref.dones, ro.dones[:T].cpu().numpy())
        return
    ro, _ = run_gpu(w, BF16, T, n_envs=n_envs, params=params, flags=flags)
    check_against_oracle(w, ro, params, T, BF16, wl.sample_env_ids(n_envs, 3, 3, 3, seed=grid))


# ---- full-size configs in the launch configuration the benchmark times ------------------------

@pytest.mark.parametrize("idx", [0, 1, 2, 3, 4])
def test_full_size_configs(idx):
    """Every workload at its full size, in bf16 with default flags (the launch shape the benchmark times).  Environment
    arrays: all environments.  Network, sampler and log-probabilities: the first 64, the last 64 and 128 seeded-random
    environments at every step, against the float64 oracle (2e-2) and against the oracle with bf16-rounded operands
    (2e-3, which also sets the margin of the action rule)."""
    w = wl.workload(idx)
    precision = _precision(w) if _tc_available(w) else FP32
    params = wl.make_params(w)
    T, E = w["T"], w["n_envs"]
    ro, _ = run_gpu(w, precision, T, params=params)
    ids = wl.sample_env_ids(E, 64, 64, 128, seed=idx)
    out = check_against_oracle(w, ro, params, T, precision, ids, obs_env_ids=None if E <= 256 else ids)
    print(idx, precision, len(ids), out)


# ---- hand-worked transitions through set_state + forced actions -------------------------------

def test_hand_worked_steps_on_the_gpu():
    import torch

    w = wl.workload(0)
    cfg = binding.make_config(w, precision=FP32, max_T=1, n_envs=6)
    ro = binding.Rollout(cfg)
    params = torch.from_numpy(wl.make_params(w)).cuda()
    far = [7, 7, 1, 7, 0, 1]
    # record: a0(r,c,l) a1(r,c,l) f0(r,c,l) f1(r,c,l) step episode total
    states = np.array([
        [2, 2, 1, 2, 4, 1, *far, 0, 0, 2],             # head-on to the same cell
        [2, 2, 1, 2, 3, 1, *far, 0, 0, 2],             # follow into a vacated cell
        [0, 5, 1, 5, 5, 1, *far, 0, 0, 2],             # wall
        [3, 2, 1, 2, 3, 2, 3, 3, 3, 6, 6, 2, 0, 0, 5],  # joint load collects level 3 of 5
        [3, 2, 1, 2, 3, 1, 3, 3, 1, 6, 6, 2, 0, 0, 3],  # collected food still blocks this step
        [3, 2, 1, 6, 6, 1, *far, 49, 0, 2],            # cap
    ], dtype=np.int32)
    acts = np.array([[4, 3], [4, 4], [1, 0], [5, 5], [5, 2], [0, 0]], dtype=np.int32)[None]
    ro.set_state(states)
    ro.run_forced(params, 1, torch.from_numpy(acts).cuda())
    assert ro.status() == 0
    after = ro.get_state()
    assert after[0, :6].tolist() == [2, 2, 1, 2, 4, 1]
    assert after[1, :6].tolist() == [2, 2, 1, 2, 4, 1]
    assert after[2, :3].tolist() == [0, 5, 1]
    assert after[3, 8] == 0 and after[3, 11] == 2
    assert after[4, 8] == 0 and after[4, 3:5].tolist() == [2, 3]
    rew = ro.rewards[0].cpu().numpy()
    assert rew[3].tolist() == [np.float32(3) / np.float32(5)] * 2
    assert rew[4].tolist() == [np.float32(1) / np.float32(3)] * 2
    assert ro.dones[0].cpu().numpy().tolist() == [0, 0, 0, 0, 0, 1]
    assert after[5, 12:14].tolist() == [0, 1]  # fresh episode 1
    fresh = oracle.env_reset(oracle.make_config(w), w["seed"], 5, 1)
    assert after[5, :2].tolist() == [fresh.agent_r[0], fresh.agent_c[0]]


# ---- determinism, continuation, reset ------------------------------------------------------------

def test_two_runs_give_identical_bytes_and_reset_replays():
    import torch

    w = wl.workload(2)
    T = 50
    cfg = binding.make_config(w, precision=FP32, max_T=T, n_envs=95)
    ro = binding.Rollout(cfg)
    params = torch.from_numpy(wl.make_params(w)).cuda()
    ro.run(params, T)
    first = [t.clone() for t in (ro.obs, ro.actions, ro.logp, ro.values, ro.rewards, ro.dones)]
    ro.reset(w["seed"])
    ro.run(params, T)
    for a, b in zip(first, (ro.obs, ro.actions, ro.logp, ro.values, ro.rewards, ro.dones)):
        assert torch.equal(a, b)
    assert ro.status() == 0


def test_two_calls_continue_like_one():
    import torch

    w = wl.workload(1)
    cfg = binding.make_config(w, precision=FP32, max_T=70, n_envs=40)
    params = torch.from_numpy(wl.make_params(w)).cuda()
    a = binding.Rollout(cfg)
    a.run(params, 70)
    b = binding.Rollout(cfg)
    b.run(params, 30)
    obs1, act1 = b.obs[:30].clone(), b.actions[:30].clone()
    b.run(params, 40)
    assert torch.equal(a.obs[:30], obs1) and torch.equal(a.actions[:30], act1)
    assert torch.equal(a.obs[30:70], b.obs[:40]) and torch.equal(a.actions[30:70], b.actions[:40])
    assert torch.equal(a.values[70], b.values[40])
    assert np.array_equal(a.get_state(), b.get_state())


def test_capacity_and_argument_errors():
    import torch

    w = wl.workload(0)
    cfg = binding.make_config(w, precision=FP32, max_T=8)
    ro = binding.Rollout(cfg, with_gae=False)
    params = torch.from_numpy(wl.make_params(w)).cuda()
    with pytest.raises(binding.MavaError) as e:
        ro.run(params, 9)
    assert e.value.code == binding.MAVA_ERR_CAPACITY
    with pytest.raises(binding.MavaError) as e:
        ro.gae(0.99, 0.95)  # no run yet and no adv/ret buffers
    assert e.value.code == binding.MAVA_ERR_INVALID_ARG
    ro.run(params, 8)
    assert ro.status() == 0 and ro.launch_count() >= 3


# ---- GAE on arbitrary data, odd shapes ------------------------------------------------------------

@pytest.mark.parametrize("idx,n_envs,T", [(0, 16, 1), (0, 5, 13), (2, 47, 37), (4, 33, 64), (1, 300, 128), (3, 9, 250),
                                              (4, 2100, 37), (2, 5464, 100),  # these two take the float4 variant
                                              # the copy-engine variant (E a multiple of 16): environments that straddle
                                              # a thread's four columns and a ragged last tile, single-step last chunk,
                                              # two agents and more chunks than a warp has lanes, a long T
                                              (2, 5488, 101), (4, 2112, 37), (1, 8208, 130), (0, 8192, 200),
                                              (0, 8192, 255)])  # too long for three stages: back to the plain scan
def test_gae_on_random_trajectories(idx, n_envs, T):
    import torch

    w = wl.workload(idx)
    cfg = binding.make_config(w, precision=FP32, max_T=T, n_envs=n_envs)
    ro = binding.Rollout(cfg)
    ro.run(torch.from_numpy(wl.make_params(w)).cuda(), T)
    g = torch.Generator(device="cuda").manual_seed(idx)
    ro.values.copy_(torch.randn(ro.values.shape, generator=g, device="cuda"))
    ro.rewards.copy_(torch.rand(ro.rewards.shape, generator=g, device="cuda"))
    ro.dones.copy_((torch.rand(ro.dones.shape, generator=g, device="cuda") < 0.1).to(torch.uint8))
    for gamma, lam in [(0.99, 0.95), (1.0, 1.0), (0.9, 0.0)]:
        ro.gae(gamma, lam)
        adv, ret = oracle.gae(ro.values.cpu().numpy(), ro.rewards.cpu().numpy(), ro.dones.cpu().numpy(),
                              float(np.float32(gamma)), float(np.float32(lam)))
        ga, gr = ro.adv.cpu().numpy(), ro.ret.cpu().numpy()
        assert np.max(np.abs(ga - adv) / np.maximum(1, np.abs(adv))) <= 1e-5
        assert np.max(np.abs(gr - ret) / np.maximum(1, np.abs(ret))) <= 1e-5


@pytest.mark.parametrize("idx,n_envs,T", [(1, 33, 256), (1, 33, 257), (1, 300, 320), (3, 5, 321), (1, 8, 512), (2, 47, 513), (0, 7, 777),
                                          (1, 300, 1000), (2, 5488, 1024)])
def test_gae_on_long_trajectories(idx, n_envs, T):
    """Up to MAVA_GAE_MAX_T steps: the last length of each chunk size and the first of the next (blocks of 1024 threads with more
    than 64 registers each are refused at launch, which once was every length above 320)."""
    import torch

    w = wl.workload(idx)
    ro = binding.Rollout(binding.make_config(w, precision=BF16, max_T=T, n_envs=n_envs))
    ro.run(torch.from_numpy(wl.make_params(w)).cuda(), T)
    g = torch.Generator(device="cuda").manual_seed(T)
    ro.values.copy_(torch.randn(ro.values.shape, generator=g, device="cuda"))
    ro.rewards.copy_(torch.rand(ro.rewards.shape, generator=g, device="cuda"))
    ro.dones.copy_((torch.rand(ro.dones.shape, generator=g, device="cuda") < 0.02).to(torch.uint8))
    ro.gae(0.99, 0.95)
    assert ro.status() == binding.MAVA_OK
    adv, ret = oracle.gae(ro.values.cpu().numpy(), ro.rewards.cpu().numpy(), ro.dones.cpu().numpy(), float(np.float32(0.99)), float(np.float32(0.95)))
    assert np.max(np.abs(ro.adv.cpu().numpy() - adv) / np.maximum(1, np.abs(adv))) <= GAE_TOL
    assert np.max(np.abs(ro.ret.cpu().numpy() - ret) / np.maximum(1, np.abs(ret))) <= GAE_TOL


# ---- tensor-core path: determinism, continuation, sharding, forcing, degenerate sizes ----------

@pytest.mark.parametrize("idx,n_envs", [(1, 150), (4, 50), (3, 40)])
def test_bf16_two_calls_continue_like_one_and_runs_repeat(idx, n_envs):
    import torch

    w = wl.workload(idx)
    cfg = binding.make_config(w, precision=BF16, max_T=50, n_envs=n_envs)
    params = torch.from_numpy(wl.make_params(w, bias_scale=0.1)).cuda()
    a = binding.Rollout(cfg)
    a.run(params, 50)
    whole = [t.clone() for t in (a.obs, a.actions, a.logp, a.values, a.rewards, a.dones)]
    a.reset(w["seed"])
    a.run(params, 50)
    for x, y in zip(whole, (a.obs, a.actions, a.logp, a.values, a.rewards, a.dones)):
        assert torch.equal(x, y)  # same seed, same bytes
    b = binding.Rollout(cfg)
    b.run(params, 20)
    first = [t[:20].clone() for t in (b.obs, b.actions, b.logp, b.rewards, b.dones)]
    b.run(params, 30)
    for x, y, z in zip(first, (b.obs, b.actions, b.logp, b.rewards, b.dones), (a.obs, a.actions, a.logp, a.rewards, a.dones)):
        assert torch.equal(z[:20], x) and torch.equal(z[20:50], y[:30])
    assert torch.equal(a.values[50], b.values[30]) and np.array_equal(a.get_state(), b.get_state())
    assert a.status() == 0 and b.status() == 0


@pytest.mark.parametrize("idx", [2, 4])
def test_env_shards_reproduce_the_whole_batch_on_the_gpu(idx):
    """Two handles with first_env offsets give the bytes of one handle over all environments."""
    import torch

    w = wl.workload(idx)
    T, n = 30, 90
    params = torch.from_numpy(wl.make_params(w)).cuda()
    whole = binding.Rollout(binding.make_config(w, precision=BF16, max_T=T, n_envs=n))
    whole.run(params, T)
    cut = 37
    lo = binding.Rollout(binding.make_config(w, precision=BF16, max_T=T, n_envs=cut))
    hi = binding.Rollout(binding.make_config(w, precision=BF16, max_T=T, n_envs=n - cut, first_env=cut))
    lo.run(params, T)
    hi.run(params, T)
    for name in ("obs", "actions", "rewards", "dones", "logp", "values"):
        full = getattr(whole, name)
        assert torch.equal(full[:, :cut], getattr(lo, name)) and torch.equal(full[:, cut:], getattr(hi, name)), name


@pytest.mark.parametrize("precision", [FP32, BF16])
@pytest.mark.parametrize("idx,n_envs,T", [(0, 1, 1), (2, 1, 3), (4, 1, 2), (3, 2, 1)])
def test_degenerate_sizes(idx, n_envs, T, precision):
    w = wl.workload(idx)
    params = wl.make_params(w)
    ro, _ = run_gpu(w, precision, T, n_envs=n_envs, params=params)
    check_against_oracle(w, ro, params, T, precision, np.arange(n_envs))


def test_forced_actions_on_the_tensor_path():
    """Teacher forcing in bf16: the oracle's own free-running actions, replayed on the GPU."""
    import torch

    w = wl.workload(1)
    T, n = 40, 70
    params = wl.make_params(w)
    ocfg = oracle.make_config(w)
    free = oracle.rollout(ocfg, w["seed"], params, T, np.arange(n))
    cfg = binding.make_config(w, precision=BF16, max_T=T, n_envs=n)
    ro = binding.Rollout(cfg)
    ro.run_forced(torch.from_numpy(params).cuda(), T, torch.from_numpy(free.actions).cuda())
    assert ro.status() == 0
    assert np.array_equal(ro.actions.cpu().numpy(), free.actions)
    assert np.array_equal(ro.obs.cpu().numpy().view(np.uint32), free.obs.view(np.uint32))
    assert np.array_equal(ro.rewards.cpu().numpy(), free.rewards) and np.array_equal(ro.dones.cpu().numpy(), free.dones)
    lp = ro.logp.cpu().numpy()
    assert np.all(np.abs(lp - free.logp) <= 2e-2 * (1 + np.abs(free.logp)))


@pytest.mark.parametrize("idx,n_envs,T", [(1, 200, 41), (2, 900, 64), (3, 60, 33), (0, 16, 5), (4, 80, 24)])
def test_collect_host_delivers_the_bytes_of_run_and_gae(idx, n_envs, T):
    """The host-buffer call (parameters in, whole trajectory out, rolled out in pieces whose copies
    overlap the kernels) against run + gae on a second handle: every array bit for bit, twice in a row."""
    import torch

    w = wl.workload(idx)
    flags = binding.MAVA_FLAG_WRITE_LOGITS
    params = torch.from_numpy(wl.make_params(w, bias_scale=0.1))
    a = binding.Rollout(binding.make_config(w, precision=BF16, max_T=T, n_envs=n_envs, flags=flags))
    b = binding.Rollout(binding.make_config(w, precision=BF16, max_T=T, n_envs=n_envs, flags=flags))
    names = ("obs", "actions", "logp", "values", "rewards", "dones", "adv", "ret", "logits")
    out = {n: torch.empty_like(getattr(b, n), device="cpu").pin_memory() for n in names}
    p_dev = params.cuda()
    for _ in range(2):
        a.run(p_dev, T)
        a.gae(wl.GAMMA, wl.LAMBDA)
        b.collect_host(params.pin_memory(), T, wl.GAMMA, wl.LAMBDA, out)
        for n in names:
            rows = T + 1 if n == "values" else T
            assert torch.equal(out[n][:rows], getattr(a, n)[:rows].cpu()), n
    assert np.array_equal(a.get_state(), b.get_state())
    assert a.status() == 0 and b.status() == 0


@pytest.mark.parametrize("name,n_envs,T,precision", [
    # one kernel form each: few rows (padded and not), 128 rows, two and three robots, recurrent, fp32
    ("cfg0_tiny_8x8_2p2f_h64", 3, 10, BF16), ("cfg1_8x8_2p2f_h128", 201, 10, BF16), ("cfg1_8x8_2p2f_h128", 2401, 10, BF16),
    ("wh0_tiny_8x8_2r2s_h64", 2399, 11, BF16), ("rec1_8x8_2p2f_gru64", 5, 10, BF16), ("rec1_8x8_2p2f_gru64", 301, 13, BF16),
    ("cfg0_tiny_8x8_2p2f_h64", 7, 10, FP32), ("rec1_8x8_2p2f_gru64", 3, 10, FP32),
    # three agents, 80 features: every piece starts on a boundary whatever the batch
    ("cfg2_10x10_3p3f_h128", 7, 11, BF16)])
def test_collect_host_where_a_piece_starts_off_a_16_byte_boundary(name, n_envs, T, precision):
    """Two agents have 79 features, so after an odd number of steps of an odd number of environments the next row is 8 bytes
    past a 16-byte boundary, where neither a bulk copy nor a 16-byte store may start (T = 10 is cut at steps 2, 5 and 7)."""
    import torch

    w = wl.workload(name)
    if w["n_agents"] == 2:  # what the case is about
        assert any((T * c // 4) * n_envs * w["n_agents"] * wl.obs_dim(w) % 4 for c in range(1, 4))
    params = torch.from_numpy(wl.make_params(w, bias_scale=0.1))
    cfg = binding.make_config(w, precision=precision, max_T=T, n_envs=n_envs, flags=binding.MAVA_FLAG_WRITE_LOGITS)
    a, b = binding.Rollout(cfg), binding.Rollout(cfg)
    names = ("obs", "actions", "logp", "values", "rewards", "dones", "adv", "ret", "logits")
    out = {n: torch.empty_like(getattr(b, n), device="cpu").pin_memory() for n in names}
    a.run(params.cuda(), T)
    a.gae(wl.GAMMA, wl.LAMBDA)
    b.collect_host(params.pin_memory(), T, wl.GAMMA, wl.LAMBDA, out)
    for n in names:
        rows = T + 1 if n == "values" else T
        assert torch.equal(out[n][:rows], getattr(a, n)[:rows].cpu()), n
    assert np.array_equal(a.get_state(), b.get_state())
    assert a.status() == 0 and b.status() == 0


@pytest.mark.parametrize("work,shapes", [("gae", [(2, BF16, 5488, 40), (2, BF16, 5488, 101), (1, BF16, 8208, 64)]),
                                         ("grad", [(3, FP32, 8, 4), (4, FP32, 8, 4), (1, FP32, 8, 4)])])
def test_handles_in_threads_of_their_own(work, shapes):
    """Handles of different shapes, each with a stream and a host thread of its own, that share kernels: every call is
    accepted and leaves the bytes that the handle leaves alone.  (The largest shared-memory size a kernel may be launched
    with belongs to the kernel: set to each launch's own need, one thread's launch was refused after another's setting.)"""
    import ctypes as C
    import threading

    import torch

    lib, hp, jobs, keep = binding.lib(), binding.ppo_defaults(), [], []
    for idx, precision, n_envs, T in shapes:
        w = wl.workload(idx)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            ro = binding.Rollout(binding.make_config(w, precision=precision, max_T=T, n_envs=n_envs))
            p = torch.from_numpy(wl.make_params(w)).cuda()
            ro.run(p, T)
            ro.gae(wl.GAMMA, wl.LAMBDA)
            grad = torch.zeros_like(p)
        if work == "gae":
            def job(ro=ro):
                return lib.mava_gae(ro.handle, wl.GAMMA, wl.LAMBDA)
            out = ro.adv
        else:
            def job(ro=ro, p=p, grad=grad):
                return lib.mava_ppo_grad(ro.handle, p.data_ptr(), C.byref(hp), grad.data_ptr(), None)
            out = grad
        assert job() == binding.MAVA_OK
        torch.cuda.synchronize()
        keep.append((ro, p, out, out.clone()))
        jobs.append(job)
    refused = [0] * len(jobs)
    start = threading.Barrier(len(jobs))

    def many(i):
        start.wait()
        for _ in range(1000):
            refused[i] += jobs[i]() != binding.MAVA_OK

    threads = [threading.Thread(target=many, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert refused == [0] * len(jobs)
    for ro, _, out, alone in keep:
        assert ro.status() == binding.MAVA_OK and torch.equal(out, alone)
        ro.close()
