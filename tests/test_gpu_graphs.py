"""Step calls recorded into a CUDA graph and replayed: the launches must not depend on what the host did between recording and
replay, in particular not on the env order that a recorded short launch reuses from an earlier one."""
import numpy as np
import pytest

from oracle import k2d_ref
from paper_2410_23208_b200 import k2d, scenes
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size,lanes,n_envs,n_steps,reuses", [("S", 8, 12700, 1, True), ("S", 8, 12700, 8, False), ("M", 32, 4500, 2, True), ("L", 0, 64, 3, False)])
def test_a_recorded_step_follows_a_reset_with_other_levels(size, lanes, n_envs, n_steps, reuses):
    import torch
    n_levels = n_envs + 500 if reuses else 64         # level ids beyond the envs: none of them may be taken for an env
    base = scenes.make_levels(size, 64, 95, static_prob=0.1)
    lv = {k: np.concatenate([v] * (-(-n_levels // 64)))[:n_levels] for k, v in base.items()}
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        env = k2d.Env(lv, n_envs, lanes_per_scene=lanes, auto_reset=1, stream=stream)
        ref = k2d_ref.RefSim(lv, n_envs, auto_reset=1, broadphase=0)
        act = scenes.make_actions(n_steps, n_envs, env.n_actions, 95)
        dev = torch.from_numpy(act).cuda()
        env.step(dev)                                 # sorts the envs where there are more than the device holds scene groups
        assert reuses == (env.resident_groups < n_envs and env.step_launches(n_steps) == 1)
        reward = torch.empty((n_steps, n_envs), dtype=torch.float32, device="cuda")
        done = torch.empty((n_steps, n_envs), dtype=torch.uint8, device="cuda")
        obs = torch.empty((n_envs, env.obs_floats), dtype=torch.float32, device="cuda")
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            env.step(dev, reward, done)
            env.obs(obs)
        ids = ((np.arange(n_envs) * 7 + n_levels - n_envs) % n_levels).astype(np.int32)
        for level_ids in (ids, None):
            env.reset(level_ids)
            ref.reset(level_ids)
            for _ in range(3):
                graph.replay()
                rr, dr = ref.step(act, n_threads=8)
            stream.synchronize()
            assert np.array_equal(reward.cpu().numpy(), rr) and np.array_equal(done.cpu().numpy(), dr)
            assert np.array_equal(obs.cpu().numpy().view(np.uint32), ref.obs().view(np.uint32))
            err, exact = parity.errors(env, ref)
            assert exact, err
            assert env.status()[3] == 3 * n_steps * n_envs      # every env once per step
        del graph
