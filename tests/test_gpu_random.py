"""Seeded random configurations against the oracle, bit for bit: what the tests by feature combine by hand is combined here at
random — scene dimensions, lanes per scene, piles, friction, masses, angles beyond the sine's range, joint kinds, resets, frame
skip, batch sizes, solver iterations, the checked build."""
import random

import numpy as np
import pytest

from paper_2410_23208_b200 import k2d, scenes
from tests import parity

pytestmark = pytest.mark.gpu


def _scenes(rng, n_levels):
    if rng.random() < 0.5:
        dims = scenes.SIZES[rng.choice("SML")]
    else:
        p, c = rng.randint(4, 12), rng.randint(0, 4)
        dims = scenes.SceneDims(p, c, rng.randint(0, min(6, p + c - 3)), rng.randint(0, 2))
    lv = scenes.make_levels(dims, n_levels, rng.randint(0, 1 << 20), static_prob=rng.choice([0.0, 0.1, 0.4]), triangle_prob=rng.choice([0.0, 0.3, 1.0]),
                            fixed_prob=rng.choice([0.0, 0.0, 0.3]), limit_prob=rng.choice([0.0, 0.0, 0.4]))
    what = rng.random()
    if what < 0.25:              # piles
        lv["pos"][:, 1:dims.n_shapes] *= np.float32(rng.choice([0.2, 0.4, 0.6]))
    elif what < 0.4:
        lv["friction"][:] = rng.choice([0.0, 1e-12, 5.0, 2e18])
    elif what < 0.5:             # masses beyond the branch-free quotients among them
        lv["density"][:] *= np.float32(10.0 ** rng.randint(-15, 9))
    elif what < 0.55:            # angles up to and beyond the sine's range
        lv["angle"][:, 1] = rng.choice([2e6, 9e5, -1e5])
    return lv


@pytest.mark.parametrize("seed", range(48))
def test_random_configuration_matches_the_oracle(seed):
    import torch
    rng = random.Random(seed)
    n_envs, n_steps, skip = rng.choice([1, 3, 7, 33, 64, 130]), rng.choice([1, 2, 9, 24]), rng.choice([1, 1, 2, 3])
    lv = _scenes(rng, min(n_envs, 24))
    env, ref = parity.make_pair(
        lv, n_envs, broadphase=rng.randint(0, 1), lanes_per_scene=rng.choice([0, 8, 16, 32]), auto_reset=rng.choice([0, 1, 2]), seed=seed,
        max_episode_steps=rng.choice([0, 5, 23]), frame_skip=skip, solver_batch=rng.choice([0, 0, 0, 1, 4, 16, 64]),
        solver_iters=rng.choice([0, 1, 4, 8, 8, 8]), warm_start=rng.choice([1, 1, 1, 0]), contact_beta=rng.choice([0.1, 0.1, 0.0]),
        joint_beta=rng.choice([0.1, 0.1, 0.0]), dense_kappa=rng.choice([0.0, 0.0, 0.2]), max_fused_steps=64, checked=rng.random() < 0.3)
    act = scenes.make_actions(-(-n_steps // skip), n_envs, env.n_actions, seed + 1) * np.float32(1.3)
    for _ in range(2):           # the second call starts from the accumulated impulses that the first one left
        want_r, want_d = ref.step(act, n_steps=n_steps, n_threads=4)
        r, d = env.step(torch.from_numpy(act).cuda(), n_steps=n_steps)
        assert np.array_equal(d.cpu().numpy(), want_d) and np.array_equal(r.cpu().numpy().view(np.uint32), want_r.view(np.uint32))
    finite = ref.status == 0     # what the words of a frozen scene hold is not specified
    st = env.get_state()
    for k in parity.STATE_KEYS:
        assert np.array_equal(st[k][finite].view(np.uint32), np.ascontiguousarray(getattr(ref, k)[finite]).view(np.uint32)), k
    for k in parity.META_KEYS:
        assert np.array_equal(st[k], getattr(ref, k)), k
    # (an angle beyond the sine's range is seen as no number, whose bits are not specified)
    rows, want = env.obs().cpu().numpy()[finite], ref.obs()[finite]
    assert np.array_equal(np.isnan(rows), np.isnan(want))
    assert np.array_equal(np.nan_to_num(rows).view(np.uint32), np.nan_to_num(want).view(np.uint32))
    if finite.all():
        assert parity.counters_match(env, ref)
