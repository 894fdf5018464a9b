"""An Env on a stream of its own: whose stream the device memory belongs to that the binding allocates, and results."""
import numpy as np
import pytest

from oracle import k2d_ref
from paper_2410_23208_b200 import k2d, scenes

pytestmark = pytest.mark.gpu


def _owner(t):
    """the stream the caching allocator holds the tensor's memory for"""
    import torch
    for seg in torch.cuda.memory_snapshot():
        if seg["address"] <= t.data_ptr() < seg["address"] + seg["total_size"]:
            return seg["stream"]
    raise AssertionError("not the allocator's memory")


@pytest.mark.parametrize("own_stream", [False, True])
def test_what_an_env_allocates_belongs_to_its_stream(own_stream):
    # A block that belongs to another stream may still be read or written there by work that is under way when the allocator
    # hands it out, and is handed out again while the Env's stream still uses it.
    import torch
    n_envs = 40
    stream = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
    lv = scenes.make_levels("M", n_envs, 33)
    env = k2d.Env(lv, n_envs, stream=stream)
    ref = k2d_ref.RefSim(lv, n_envs, broadphase=0)
    act = scenes.make_actions(6, n_envs, env.n_actions, 33)
    dev = torch.from_numpy(act).cuda()
    torch.cuda.synchronize()
    r, d = env.step(dev[:3])
    r2, d2, o = env.step_obs(dev[3:])
    o2, img, trace = env.obs(), env.render(), env.enable_trace()
    torch.cuda.synchronize()
    for t in (env.state_buf, env.level_buf, r, d, r2, d2, o, o2, img, trace):
        assert _owner(t) == stream.cuda_stream
    rr, dr = ref.step(act)
    assert np.array_equal(torch.cat([r, r2]).cpu().numpy(), rr) and np.array_equal(torch.cat([d, d2]).cpu().numpy(), dr)
    assert torch.equal(o, o2) and np.array_equal(o.cpu().numpy().view(np.uint32), ref.obs().view(np.uint32))
