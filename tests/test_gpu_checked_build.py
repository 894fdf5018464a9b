"""The checked build of the library (-DK2D_CHECKED: every index the kernels unpack from packed words or read from tables is
compared with its limit, a violation sets a status bit and the access is redirected; nothing traps) run over the cases that
use the most index arithmetic: the three size classes, every lanes-per-scene setting, piles that overflow the on-chip
records, auto-reset from a pool, more envs than resident groups, the batched solve, the fused observation.  It stands in for
a memory checker: results must still equal the oracle's and no check may fire."""
import numpy as np
import pytest

from paper_2410_23208_b200 import k2d, scenes
from tests import parity


def test_checked_library_builds_and_says_so():
    lib = k2d.load_library(checked=True)
    assert lib.k2d_is_checked_build() == 1 and k2d.load_library().k2d_is_checked_build() == 0
    for name in k2d.EXPORTS:
        assert hasattr(lib, name), name


def _pair(lv, n_envs, **cfg):
    env, ref = parity.make_pair(lv, n_envs, checked=True, **cfg)
    assert env.lib.k2d_is_checked_build() == 1
    return env, ref


def _run(env, ref, act, chunk):
    (r, d), (rr, dr) = parity.step_both(env, ref, act, chunk=chunk, n_threads=8)
    assert np.array_equal(r, rr) and np.array_equal(d, dr)
    err, exact = parity.errors(env, ref)
    assert exact, err
    assert parity.counters_match(env, ref)          # k2d_status raises if an index check fired


@pytest.mark.gpu
@pytest.mark.parametrize("size,n_envs,lanes", [("S", 40, 8), ("S", 40, 0), ("M", 48, 16), ("M", 48, 32), ("L", 72, 8), ("L", 72, 16), ("L", 72, 32)])
def test_no_index_check_fires_on_generated_scenes(size, n_envs, lanes):
    lv = scenes.make_levels(size, n_envs, 17, static_prob=0.1, triangle_prob=0.2, fixed_prob=0.2, limit_prob=0.2)
    lv["pos"][: n_envs // 6, 1:, 0] *= 0.15            # some crowded scenes: second records and the memory-record path
    env, ref = _pair(lv, n_envs, lanes_per_scene=lanes, auto_reset=2, max_episode_steps=17, seed=4, dense_kappa=0.1)
    _run(env, ref, scenes.make_actions(60, n_envs, env.n_actions, 17), 13)
    import torch
    r, d, o = env.step_obs(torch.zeros((1, n_envs, env.n_actions), device="cuda"))
    ref.step(np.zeros((1, n_envs, env.n_actions), np.float32))
    assert np.array_equal(o.cpu().numpy().view(np.uint32), ref.obs().view(np.uint32))
    env.status()


@pytest.mark.gpu
@pytest.mark.parametrize("lanes", [8, 16, 32])
def test_no_index_check_fires_on_piles(lanes):
    lv = scenes.make_levels("L", 6, 51)
    rng = np.random.default_rng(51)
    lv["pos"][:, 1:, 0] = rng.uniform(-0.3, 0.3, (6, 15)).astype(np.float32)
    lv["pos"][:, 1:, 1] = rng.uniform(0.8, 1.4, (6, 15)).astype(np.float32)
    lv["joint_active"][:] = 0
    env, ref = _pair(lv, 6, lanes_per_scene=lanes)
    _run(env, ref, scenes.make_actions(16, 6, env.n_actions, 51), 4)


@pytest.mark.gpu
def test_no_index_check_fires_through_the_work_queue_and_in_the_batched_solve():
    lv = scenes.make_levels("L", 256, 77, static_prob=0.1)
    for n_envs, lanes in ((9600, 8), (6200, 16)):
        env, ref = _pair(lv, n_envs, auto_reset=2, max_episode_steps=10, seed=77, max_fused_steps=24, lanes_per_scene=lanes)
        assert env.resident_groups < n_envs
        _run(env, ref, scenes.make_actions(20, n_envs, env.n_actions, 77), 20)
    lv = scenes.make_levels("M", 64, 78, static_prob=0.1)
    lv["pos"][:16, 1:, 0] *= 0.15
    env, ref = _pair(lv, 64, solver_batch=16)
    _run(env, ref, scenes.make_actions(30, 64, env.n_actions, 78), 10)


@pytest.mark.gpu
def test_a_bad_count_in_the_state_record_is_caught_and_redirected():
    # the number of warm entries of env 0 is overwritten with 1000 from the host (far beyond the 21 pairs of an S scene); the
    # checked build reports it through k2d_status and uses 0 instead, so nothing is read out of range; k2d_reset clears it
    import torch
    n_envs = 8
    lv = scenes.make_levels("S", n_envs, 3)
    env = k2d.Env(lv, n_envs, checked=True)
    act = torch.zeros((4, n_envs, env.n_actions), device="cuda")
    env.step(act)
    env.status()
    # state buffer: 4096-byte control block, then level ids and chunk counters (4 bytes per env each, 256-byte aligned), then
    # the env records; an S record has its meta words after 6 x 7 body words and 3 joint words, the count is meta word 4
    offset = 4096 + 512 + 4 * (6 * 7 + 3 + 4)
    assert int(env.state_buf[offset:offset + 4].view(torch.int32)[0]) <= 21
    env.state_buf[offset:offset + 4].view(torch.int32)[0] = 1000
    torch.cuda.synchronize()
    env.step(act)
    torch.cuda.synchronize()
    with pytest.raises(k2d.K2DError, match="index check"):
        env.status()
    env.reset()
    env.step(act)
    assert env.status()[3] == 4 * n_envs


# S scenes: words of a level record (joint, thruster, the dense reward's shapes) and of a state record (level id), in bytes from
# the start of their buffer, and what is planted there
PLANTED = {
    "joint": ("level_buf", 4 * 188, 0xff, 200),
    "thruster": ("level_buf", 4 * 200, 0xff, 200),
    "first green shape": ("level_buf", 4 * 215, 0xff, 250),
    "level id": ("state_buf", 4096 + 512 + 4 * (6 * 7 + 3 + 2), 0xffffffff, 99999),
}


@pytest.mark.gpu
@pytest.mark.parametrize("what,call", [(w, c) for w in ("joint", "thruster", "level id") for c in ("step", "step_obs", "obs")] +
                         [("first green shape", "step"), ("level id", "render"), ("level id", "reset inside the step")])
def test_a_bad_index_in_a_level_or_state_record_is_caught_and_redirected(what, call):
    # checked build only: the word is wrong in the caller's own buffer, every use of it is compared with its limit and redirected
    import torch
    n_envs = 8
    lv = scenes.make_levels("S", n_envs, 3)
    env = k2d.Env(lv, n_envs, checked=True, dense_kappa=0.1, auto_reset=1, max_episode_steps=2 if "reset" in call else 0)
    assert (env.cfg.n_polygons, env.cfg.n_circles, env.cfg.n_joints, env.cfg.n_thrusters) == (5, 2, 1, 1)
    act = torch.zeros((4, n_envs, env.n_actions), device="cuda")

    def run():
        if call == "step_obs":
            env.step_obs(act)
        elif call in ("obs", "render"):
            getattr(env, call)()
        else:
            env.step(act)
        torch.cuda.synchronize()

    run()
    env.status()
    name, at, mask, value = PLANTED[what]
    word = getattr(env, name)[at:at + 4].view(torch.int32)
    good = int(word[0])
    new = (good & 0xffffffff & ~mask) | value
    word[0] = new - (1 << 32) if new >= 1 << 31 else new
    torch.cuda.synchronize()
    run()
    with pytest.raises(k2d.K2DError, match="index check"):
        env.status()
    word[0] = good
    env.reset()
    run()
    env.status()


# ---------------------------------------------------------------- the build that counts cycles per phase of a step
def test_phase_clock_library_builds_and_the_plain_library_refuses_the_call():
    from paper_2410_23208_b200 import build
    lib = k2d.load_library(phase_clocks=True)
    assert build.LIB_PHASES.endswith("libk2d_phases.so") and lib.k2d_is_checked_build() == 0
    assert len(k2d.PHASES) == 14


@pytest.mark.gpu
def test_phase_clocks_count_every_phase_and_change_no_result():
    n_envs = 96
    lv = scenes.make_levels("L", 48, 77, static_prob=0.1)
    lv["pos"][:8, 1:, 0] *= 0.2                          # some crowded scenes: the memory-record path is timed too
    env, ref = parity.make_pair(lv, n_envs, phase_clocks=True, lanes_per_scene=16, auto_reset=2, max_episode_steps=12, seed=5)
    act = scenes.make_actions(24, n_envs, env.n_actions, 77)
    (r, d), (rr, dr) = parity.step_both(env, ref, act, chunk=24)
    assert np.array_equal(r.view(np.uint32), rr.view(np.uint32)) and np.array_equal(d, dr)
    err, exact = parity.errors(env, ref)
    assert exact, err
    cycles = env.phase_cycles()
    assert set(cycles) == set(k2d.PHASES)
    for name in ("geometry", "box_test", "narrowphase", "records", "iterations", "integrate_correct", "epilogue", "load", "store"):
        assert cycles[name] > 0, name
    assert cycles["iterations"] > cycles["joint_prestep"]
    assert sum(env.phase_cycles().values()) == 0             # reading clears the sums
    # the library proper has no counters
    plain = k2d.Env(lv, 8)
    with pytest.raises(k2d.K2DError, match="build"):
        plain.phase_cycles()


@pytest.mark.gpu
@pytest.mark.parametrize("size,lanes", [("S", 16), ("M", 8), ("L", 8), ("L", 16)])
def test_frozen_scenes_do_not_send_their_neighbours_through_the_compared_axes(size, lanes):
    """a scene that is frozen (its words are no numbers) and the empty groups of a last, partly filled warp leave the path of the
    other scenes of a warp alone; a scene that is stepped at such coordinates does not"""
    import torch
    n_envs = 41
    lv = scenes.make_levels(size, n_envs, 78, static_prob=0.1)
    env, other = (k2d.Env(lv, n_envs, phase_clocks=True, lanes_per_scene=lanes) for _ in range(2))
    act = torch.from_numpy(scenes.make_actions(12, n_envs, env.n_actions, 78)).cuda()
    frozen = np.arange(n_envs) % 4 == 1
    st = env.get_state()
    st["pos"][frozen] = np.nan
    st["status"][frozen] = 1
    env.set_state(st)
    env.slow_paths()
    reward, done = env.step(act)
    assert env.slow_paths()["axes"] == 0
    want_r, want_d = other.step(act)
    keep = torch.from_numpy(~frozen).cuda()
    assert torch.equal(reward[:, keep], want_r[:, keep]) and torch.equal(done[:, keep], want_d[:, keep])
    assert bool((done[:, ~keep] == 1).all()) and bool((reward[:, ~keep] == 0).all())
    got, want = env.get_state(), other.get_state()
    for k in parity.STATE_KEYS:
        assert np.array_equal(got[k][~frozen].view(np.uint32), want[k][~frozen].view(np.uint32)), k
    st = other.get_state()
    st["pos"][7, 1] = 3.0e18
    other.set_state(st)
    other.slow_paths()
    other.step(act)
    assert 0 < other.slow_paths()["axes"] <= 12 and other.slow_paths()["axes"] == 0      # one warp of the launch; reading clears
    plain = k2d.Env(lv, 8)
    with pytest.raises(k2d.K2DError, match="build"):
        plain.slow_paths()


@pytest.mark.gpu
@pytest.mark.parametrize("size,lanes", [("S", 32), ("M", 8), ("L", 8), ("L", 16)])
def test_constants_of_zero_are_ordinary_operands(size, lanes):
    """with the positional corrections switched off and no friction, joint rows and contact records take the branch-free quotients
    and roots as ever; masses beyond their range do not"""
    n_envs = 40
    lv = scenes.make_levels(size, n_envs, 79, static_prob=0.1)
    lv["friction"][:] = 0.0
    env, ref = parity.make_pair(lv, n_envs, phase_clocks=True, lanes_per_scene=lanes, joint_beta=0.0, contact_beta=0.0, joint_alpha=0.0, slop=0.0)
    act = scenes.make_actions(30, n_envs, env.n_actions, 79)
    env.slow_paths()
    (r, d), (rr, dr) = parity.step_both(env, ref, act)
    assert env.slow_paths() == {"axes": 0, "joint_rows": 0, "records": 0}
    assert np.array_equal(r, rr) and np.array_equal(d, dr) and ref.counters[2] > 0 and parity.errors(env, ref)[1]
    for k in ("density", "motor_power", "thr_power"):
        lv[k][:] *= np.float32(1e-21)
    env, ref = parity.make_pair(lv, n_envs, phase_clocks=True, lanes_per_scene=lanes)
    env.slow_paths()
    (r, d), (rr, dr) = parity.step_both(env, ref, np.zeros_like(act))
    slow = env.slow_paths()
    assert slow["joint_rows"] > 0 and slow["records"] > 0 and parity.errors(env, ref)[1]
