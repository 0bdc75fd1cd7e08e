"""The give-up path of the kernels' bounded waits, exercised without faulting, trapping or hanging anything: one armed
launch makes one thread block wait briefly on a barrier phase that nothing completes, at a point where none of its
MMAs is outstanding (and no copy but the update's weight image).  The block must record the time-out and leave in order (copies drained, tensor memory
freed, its partner thread group walked through the hand-over protocol), the status call must report it once, and the
same handle must work again afterwards."""
import numpy as np
import pytest

from paper_2107_01460_b200 import binding, workloads as wl

from parity import check_against_oracle

pytestmark = pytest.mark.gpu
BF16 = binding.MAVA_PRECISION_BF16


def _fresh_run_matches(w, ro, params, p_dev, T, ids):
    ro.reset(w["seed"])
    ro.run(p_dev, T)
    ro.gae(np.float32(wl.GAMMA), np.float32(wl.LAMBDA))
    assert ro.status() == binding.MAVA_OK
    check_against_oracle(w, ro, params, T, BF16, ids)


def test_gae_copy_engine_kernel_gives_up_and_recovers():
    import torch

    w = wl.workload(2)
    T, n_envs = 32, 5488  # 16 464 columns: the persistent copy-engine kernel
    params = wl.make_params(w)
    ro = binding.Rollout(binding.make_config(w, precision=BF16, max_T=T, n_envs=n_envs, flags=binding.MAVA_FLAG_WRITE_LOGITS))
    p_dev = torch.from_numpy(params).cuda()
    ro.run(p_dev, T)
    ro.debug_expire_next_wait(binding.MAVA_EXPIRE_GAE)
    ro.gae(wl.GAMMA, wl.LAMBDA)
    assert ro.status() == binding.MAVA_ERR_DEVICE_TIMEOUT
    assert ro.status() == binding.MAVA_OK  # reported once
    _fresh_run_matches(w, ro, params, p_dev, T, wl.sample_env_ids(n_envs, 4, 4, 8, seed=7))


@pytest.mark.parametrize("idx,n_envs", [(4, 1200), (2, 5000)])
def test_rollout_kernel_gives_up_and_recovers(idx, n_envs):
    """idx 4: the two thread groups of an SM share one tile set and hand it to each other through named barriers; the
    group that gives up, and its partner once it sees the flag, must keep walking that protocol to the end.
    idx 2: independent groups; the one that gives up simply stops."""
    import torch

    w = wl.workload(idx)
    T = 24
    params = wl.make_params(w)
    ro = binding.Rollout(binding.make_config(w, precision=BF16, max_T=T, n_envs=n_envs, flags=binding.MAVA_FLAG_WRITE_LOGITS))
    p_dev = torch.from_numpy(params).cuda()
    ro.debug_expire_next_wait(binding.MAVA_EXPIRE_ROLLOUT)
    ro.run(p_dev, T)
    assert ro.status() == binding.MAVA_ERR_DEVICE_TIMEOUT
    assert ro.status() == binding.MAVA_OK
    _fresh_run_matches(w, ro, params, p_dev, T, wl.sample_env_ids(n_envs, 4, 4, 8, seed=7))


@pytest.mark.parametrize("idx,n_envs,T", [(0, 24, 16), (2, 395, 48)])
def test_update_kernel_gives_up_and_recovers(idx, n_envs, T):
    """The warp that issues the products gives up before its first, with the second half of the weight image possibly still on
    its way: every other role of the block runs into its own limit (idx 2: three tiles per SM, so the row loaders stand
    before an x tile that nobody frees), the image lands, and the block leaves.  The same call then gives the same bytes."""
    import torch

    w = wl.workload(idx)
    ro = binding.Rollout(binding.make_config(w, precision=BF16, max_T=T, n_envs=n_envs))
    params = torch.from_numpy(wl.make_params(w)).cuda()
    ro.run(params, T)
    ro.gae(wl.GAMMA, wl.LAMBDA)
    want = [x.clone() for x in ro.ppo_grad(params)]
    assert ro.status() == binding.MAVA_OK
    ro.debug_expire_next_wait(binding.MAVA_EXPIRE_UPDATE)
    ro.ppo_grad(params)
    assert ro.status() == binding.MAVA_ERR_DEVICE_TIMEOUT
    assert ro.status() == binding.MAVA_OK
    got = ro.ppo_grad(params)
    assert ro.status() == binding.MAVA_OK
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    ro.close()


def test_gae_longer_than_its_limit_is_a_capacity_error():
    import torch

    w = wl.workload(0)
    T = binding.MAVA_GAE_MAX_T + 1
    ro = binding.Rollout(binding.make_config(w, precision=binding.MAVA_PRECISION_FP32, max_T=T, n_envs=4))
    ro.run(torch.from_numpy(wl.make_params(w)).cuda(), T)
    with pytest.raises(binding.MavaError) as e:
        ro.gae(wl.GAMMA, wl.LAMBDA)
    assert e.value.code == binding.MAVA_ERR_CAPACITY
    assert ro.status() == binding.MAVA_OK


@pytest.mark.parametrize("idx", [1, 4])
def test_a_failed_launch_leaves_no_error_behind(idx):
    """A launch that the runtime refuses on the host (into a stream capture that is no longer valid): the return code tells of it,
    and the runtime's own record, which the caller's process would take for a failure of whatever it launches next, is clear."""
    import ctypes as C

    import torch

    w = wl.workload(idx)
    T, n_envs = 8, 32
    p_dev = torch.from_numpy(wl.make_params(w)).cuda()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ro = binding.Rollout(binding.make_config(w, precision=BF16, max_T=T, n_envs=n_envs))
        ro.run(p_dev, T)
        ro.gae(wl.GAMMA, wl.LAMBDA)
    ro.ppo_grad(p_dev)
    torch.cuda.synchronize()
    want = ro.obs.clone(), ro.logp.clone()
    rt = C.CDLL("libcudart.so.12")  # the instance that the library and torch share
    s, graph = C.c_void_p(stream.cuda_stream), C.c_void_p()
    assert rt.cudaStreamBeginCapture(s, 2) == 0  # relaxed: only this stream is concerned
    assert rt.cudaStreamSynchronize(s) != 0      # not allowed while capturing: the capture is invalid from here on
    rt.cudaGetLastError()
    codes = [binding.lib().mava_rollout_run(ro.handle, p_dev.data_ptr(), T), binding.lib().mava_gae(ro.handle, 0.99, 0.95)]
    record = rt.cudaPeekAtLastError()
    assert rt.cudaStreamEndCapture(s, C.byref(graph)) != 0
    rt.cudaGetLastError()
    assert codes == [binding.MAVA_ERR_CUDA] * 2 and record == 0
    ro.reset(w["seed"])
    ro.run(p_dev, T)
    ro.gae(wl.GAMMA, wl.LAMBDA)
    assert ro.status() == binding.MAVA_OK
    assert torch.equal(ro.obs, want[0]) and torch.equal(ro.logp, want[1])
    ro.close()
