"""GPU parity at the edges of the contact solve's storage and schedule: pairs beyond the shared-memory records, beyond what a
schedule holds, more solver levels than the fast sweep takes, a pair whose second manifold alone is active, friction that is
limited by comparisons, crowded scenes in the batched solve, and env counts around the launch shapes of the step kernel."""
import numpy as np
import pytest

from paper_2410_23208_b200 import scenes
from tests import parity

pytestmark = pytest.mark.gpu


def _touching(ref):
    on = ref.manifold[:, :, 5] > 0                   # 66 polygon pairs of an L scene own two manifold slots each, the others one
    return (on[:, :132:2] | on[:, 1:132:2]).sum(1) + on[:, 132:].sum(1)


def _piles(n, seed, spread):
    lv = scenes.make_levels("L", n, seed)
    rng = np.random.default_rng(seed)
    lv["pos"][:, 1:, 0] = (rng.uniform(-1, 1, (n, 15)) * spread[:, None]).astype(np.float32)
    lv["pos"][:, 1:, 1] = (0.6 + rng.uniform(0, 1, (n, 15)) * spread[:, None]).astype(np.float32)
    return lv


def _exact(env, ref, act, chunk=None):
    (r, d), (rr, dr) = parity.step_both(env, ref, act, chunk=chunk)
    err, exact = parity.errors(env, ref)
    assert exact, err
    assert np.array_equal(r, rr) and np.array_equal(d, dr)


@pytest.mark.parametrize("lanes", [8, 16, 32])
@pytest.mark.parametrize("batch", [0, 16])
def test_scenes_around_the_record_counts(lanes, batch):
    # 20 records in shared memory with 8 lanes, 31 in a schedule: piles of growing spread have counts on every side of both
    n = 48
    lv = _piles(n, 61, np.linspace(0.3, 2.2, n))
    env, ref = parity.make_pair(lv, n, lanes_per_scene=lanes, solver_batch=batch)
    act = scenes.make_actions(10, n, env.n_actions, 61)
    seen = set()
    for k in range(10):
        _exact(env, ref, act[k:k + 1])
        seen |= set(_touching(ref).tolist())
    assert max(seen) > 31 and len(seen & set(range(21, 32))) >= 5 and len(seen & set(range(9, 21))) >= 5


@pytest.mark.parametrize("lanes", [8, 16, 32])
@pytest.mark.parametrize("height", [7, 8, 9, 15])
def test_towers_with_as_many_levels_as_boxes(lanes, height):
    # a tower is one chain of contacts: as many solver levels as bodies (the fast sweep takes 8)
    dims = scenes.SIZES["L"]
    polys = [dict(half=(5.0, 0.5), pos=(0.0, -0.5), static=1)]
    polys += [dict(half=(0.3, 0.1), pos=(0.01 * (i % 3), 0.099 + 0.199 * i)) for i in range(min(height, 11))]
    circles = [dict(radius=0.1, pos=(0.01, 0.099 + 0.199 * (11 + i))) for i in range(max(0, height - 11))]
    lv = scenes.concat_levels([scenes.custom_level(dims, polygons=polys, circles=circles)] * 3)
    env, ref = parity.make_pair(lv, 3, lanes_per_scene=lanes)
    _exact(env, ref, scenes.make_actions(12, 3, env.n_actions, 7), chunk=5)
    assert _touching(ref).max() >= height - 1


@pytest.mark.parametrize("size,lanes", [("L", 8), ("M", 16), ("S", 32)])
def test_pairs_whose_second_manifold_alone_is_active_carry_their_impulses_over(size, lanes):
    n = 96
    lv = scenes.make_levels(size, n, 63, triangle_prob=0.3)
    env, ref = parity.make_pair(lv, n, lanes_per_scene=lanes)
    act = scenes.make_actions(60, n, env.n_actions, 63)
    p = scenes.SIZES[size].n_polygons
    found = 0
    for k in range(0, 60, 4):
        _exact(env, ref, act[k:k + 4], chunk=3)
        on = ref.manifold[:, :p * (p - 1), 5] > 0
        found += int((~on[:, ::2] & on[:, 1::2]).sum())
    assert found > 0


@pytest.mark.parametrize("lanes", [8, 32])
def test_friction_too_large_for_the_fast_limit(lanes):
    lv = scenes.make_levels("M", 24, 64)
    lv["friction"][::2, 2] = 2.0e18
    env, ref = parity.make_pair(lv, 24, lanes_per_scene=lanes)
    _exact(env, ref, scenes.make_actions(40, 24, env.n_actions, 64), chunk=9)


@pytest.mark.parametrize("lanes", [8, 16, 32])
@pytest.mark.parametrize("solver_iters", [1, 8])
def test_a_normal_impulse_that_overflows_without_friction(lanes, solver_iters):
    # The friction bound of a frictionless pair is 0 x infinity once its normal impulse overflows.  The value it limits is then no
    # number either, whichever way the limit is taken; env and oracle agree on every number and on what is none.  (One pair of
    # movable shapes per scene: what an overflow does to a fixated shape, which the library never writes, is not specified.)
    dims, levels = scenes.SIZES["M"], []
    for tilt in (0.0, 0.7, -0.4):
        nx, ny = -np.sin(tilt), np.cos(tilt)
        for k, vel in enumerate(((0.0, -3.0e38), (2.0e38, -2.5e38), (-1.0e38, -3.0e38), (0.5, -1.0))):
            polys = [dict(half=(5.0, 0.5), pos=(-0.5 * nx, -0.5 * ny), angle=tilt, density=2.0, friction=0.0)]
            box = dict(half=(0.5, 0.5), pos=(0.49 * nx, 0.49 * ny), angle=tilt, vel=vel, density=2.0, friction=0.0)
            circle = dict(radius=0.8, pos=(0.79 * nx + 2.5 * ny, 0.79 * ny - 2.5 * nx), vel=vel, density=2.0, friction=0.0)
            levels.append(scenes.custom_level(dims, polygons=polys + [box]))
            levels.append(scenes.custom_level(dims, polygons=polys, circles=[circle]))
    env, ref = parity.make_pair(scenes.concat_levels(levels), 24, lanes_per_scene=lanes, solver_iters=solver_iters)
    act = scenes.make_actions(3, 24, env.n_actions, 68)
    for k in range(3):
        (r, d), (rr, dr) = parity.step_both(env, ref, act[k:k + 1])
        assert np.array_equal(r, rr) and np.array_equal(d, dr)
        st = env.get_state()
        for key in parity.STATE_KEYS:
            assert np.array_equal(st[key], getattr(ref, key), equal_nan=True), key
        for key in parity.META_KEYS:
            assert np.array_equal(st[key], getattr(ref, key)), key
    assert (ref.status[6::8] == 0).all() and (ref.status[7::8] == 0).all() and ref.status.sum() >= 12
    # a bound that was no number, and a value that was none (with one iteration they stay in the accumulated impulses)
    assert solver_iters > 1 or (np.isinf(ref.acc[:, :, 0]) & np.isnan(ref.acc[:, :, 1])).sum() >= 12


@pytest.mark.parametrize("n_envs", [7103, 7105, 9471, 9472, 9473])
def test_env_counts_around_the_launch_shapes(n_envs):
    # 48 and 64 scenes per SM on 148 SMs
    lv = scenes.make_levels("S", 64, 65, static_prob=0.1)
    env, ref = parity.make_pair(lv, n_envs, lanes_per_scene=8, auto_reset=2, max_episode_steps=7, seed=65)
    act = scenes.make_actions(11, n_envs, env.n_actions, 65)
    (r, d), (rr, dr) = parity.step_both(env, ref, act[:9], n_threads=8)
    assert np.array_equal(r, rr) and np.array_equal(d, dr)
    (r, d), (rr, dr) = parity.step_both(env, ref, act[9:], chunk=1, n_threads=8)
    err, exact = parity.errors(env, ref)
    assert exact, err


@pytest.mark.parametrize("size,n_envs,lanes", [("S", 593, 32), ("S", 1183, 32), ("S", 2368, 16), ("M", 2369, 16), ("L", 1185, 32), ("L", 4735, 16), ("S", 4737, 8), ("L", 2663, 0), ("L", 6000, 0)])
def test_block_sizes_of_launches_of_one_wave(size, n_envs, lanes):
    # one block per SM of 128, 256, 384 or 512 threads, envs on either side of a full device; one step at a time (small blocks
    # where the block would fill an SM) and several
    lv = scenes.make_levels(size, 48, 66, static_prob=0.1)
    lv["pos"][:8, 1:, 0] *= 0.3          # a few piles, whose records reach the scratch slots
    env, ref = parity.make_pair(lv, n_envs, lanes_per_scene=lanes, auto_reset=2, max_episode_steps=6, seed=66)
    assert env.resident_groups == n_envs
    act = scenes.make_actions(9, n_envs, env.n_actions, 66)
    (r, d), (rr, dr) = parity.step_both(env, ref, act[:2], chunk=1, n_threads=8)
    assert np.array_equal(r, rr) and np.array_equal(d, dr)
    (r, d), (rr, dr) = parity.step_both(env, ref, act[2:], n_threads=8)
    err, exact = parity.errors(env, ref)
    assert exact and np.array_equal(r, rr) and np.array_equal(d, dr), err


def test_state_of_scenes_without_joints():
    dims = scenes.SceneDims(6, 0, 0, 1)
    lv = scenes.make_levels(dims, 8, 67)
    env, ref = parity.make_pair(lv, 8)
    _exact(env, ref, scenes.make_actions(5, 8, env.n_actions, 67))
    env.set_state(env.get_state())
    _exact(env, ref, scenes.make_actions(5, 8, env.n_actions, 68))


@pytest.mark.parametrize("size,n_envs,lanes", [("S", 1, 32), ("S", 129, 16), ("M", 37, 16), ("L", 130, 8), ("L", 600, 0), ("S", 5003, 0), ("S", 20011, 0)])
def test_work_counters_of_blocks_of_every_fill(size, n_envs, lanes):
    """counts that leave the blocks together: one scene, blocks partly filled, several blocks, small blocks beside one another
    (one step of many envs), several waves; and launches long enough for the groups to write theirs out on the way"""
    lv = scenes.make_levels(size, min(n_envs, 64), 67, static_prob=0.1)
    env, ref = parity.make_pair(lv, n_envs, broadphase=1, lanes_per_scene=lanes, auto_reset=2, max_episode_steps=40, seed=67, max_fused_steps=300)
    for i, n_steps in enumerate([1, 1, 2] + ([300] if n_envs < 200 else [9])):
        act = scenes.make_actions(n_steps, n_envs, env.n_actions, 670 + i)
        (r, d), (rr, dr) = parity.step_both(env, ref, act, n_threads=8)
        assert np.array_equal(r, rr) and np.array_equal(d, dr)
        assert parity.counters_match(env, ref), (n_steps, env.status(), ref.counters)
    assert parity.errors(env, ref)[1]
