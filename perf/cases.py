"""What a user of the batched environment step has it do, as cases to time and to compare.

A case is one call pattern of ``paper_2410_23208_b200.k2d``: scenes of a size class (or of dimensions in between), a number
of envs, engine steps per call, continuous or multi-discrete actions, what is observed afterwards (entity rows in the same
or in a second launch, or pixels), and how finished episodes restart.  The sizes are the five workloads of
``scenes.WORKLOADS``, the paper's training set-up (frame skip 2, one decision per call) and sizes in between.

``prepare`` brings the scenes into the state a training run finds them in: they have been stepped until the piles lie on the
floor, and where episodes have a horizon the envs are at different steps of theirs.  Actions lie on the device already, as
a policy leaves them.  Results are bit-reproducible by the library's contract, so outputs are compared exactly.
"""
import math

import numpy as np
import torch

from paper_2410_23208_b200 import k2d, scenes

LARGEST = 131072 * 32          # env-steps of L scenes that one pass takes at most
NEVER, SAME_LEVEL, POOL = k2d.RESET_NONE, k2d.RESET_SAME_LEVEL, k2d.RESET_POOL


def _case(size, n_envs, n_steps, **more):
    d = scenes.SIZES[size] if isinstance(size, str) else size
    c = dict(kind="step", polygons=d.n_polygons, circles=d.n_circles, joints=d.n_joints, thrusters=d.n_thrusters,
             n_envs=n_envs, n_steps=n_steps, frame_skip=1, actions="continuous", observe="rows", reset=POOL, horizon=256,
             levels=min(n_envs, 1024), static=0.1, triangles=0.0, fixed=0.0, limited=0.0, solver_batch=0)
    c.update(more)
    return c


def listed():
    odd = scenes.SceneDims(8, 2, 3, 1)
    return [
        # a policy watched or evaluated in a few envs: one decision, one observation per call; launches and latency count
        dict(_case("S", 64, 1, observe="fused rows", reset=SAME_LEVEL, horizon=0), name="s64_act"),
        # workload 0: a whole rollout of 16 small scenes in one call, no restarts
        dict(_case("S", 16, 100, observe="rows", reset=NEVER, horizon=0, static=0.0), name="s16_rollout"),
        # workload 1: small scenes in fused rollouts, restarting on their own level
        dict(_case("S", 4096, 32, reset=SAME_LEVEL, horizon=0), name="s4096_rollout"),
        # training on medium scenes with the multi-discrete action space and the paper's frame skip: one decision per call
        dict(_case("M", 2048, 2, frame_skip=2, actions="discrete"), name="m2048_discrete"),
        # workload 2: medium scenes in fused rollouts
        dict(_case("M", 16384, 32, reset=SAME_LEVEL, horizon=0), name="m16384_rollout"),
        # scenes between the size classes, with triangles, fixed and limited joints, an odd number of envs and of steps
        dict(_case(odd, 5003, 17, triangles=0.3, fixed=0.2, limited=0.3), name="odd5003_rollout"),
        # training on pixels: one decision and one 125 x 125 image per call
        dict(_case("L", 2048, 2, frame_skip=2, observe="pixels"), name="l2048_pixels"),
        # the paper's batched contact solve at its default batch size of 16
        dict(_case("L", 4096, 8, solver_batch=16), name="l4096_batch16"),
        # training on large scenes: one decision (two engine steps) and the entity rows in one call
        dict(_case("L", 16384, 2, frame_skip=2, observe="fused rows"), name="l16384_act"),
        # workload 3, the benchmark's: large scenes in fused rollouts, restarting on levels of the pool
        dict(_case("L", 16384, 32), name="l16384_rollout"),
        # workload 4 at its largest
        dict(_case("L", 131072, 32), name="l131072_rollout"),
        # the level generator's filter: what doing nothing achieves on 1024 levels, from host arrays to host outcomes
        dict(_case("L", 1024, 256, kind="noop", reset=NEVER, horizon=0), name="noop1024"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    r = rng.random()
    if r < 0.6:
        dims = scenes.SIZES[rng.choice("SML")]
    else:
        p, c = rng.randint(4, 12), rng.randint(0, 4)
        dims = scenes.SceneDims(p, c, rng.randint(0, min(6, p + c - 3)), rng.randint(0, 2))
    kinds = dict(triangles=0.3, fixed=0.2, limited=0.3) if rng.random() < 0.25 else {}
    what = rng.random()
    if what < 0.08:
        n = _log_int(rng, 64, 1024)
        return _case(dims, n, _log_int(rng, 64, 256), kind="noop", reset=NEVER, horizon=0, **kinds)
    restart = rng.choice([dict(reset=POOL, horizon=256), dict(reset=SAME_LEVEL, horizon=0), dict(reset=POOL, horizon=rng.randint(64, 512))])
    if what < 0.16:      # pixels
        skip = rng.choice([1, 2, 4])
        return _case(dims, _log_int(rng, 64, 8192), skip, frame_skip=skip, observe="pixels", **restart, **kinds)
    if what < 0.24:      # batched contact solve
        return _case(dims, _log_int(rng, 256, 8192), _log_int(rng, 1, 16), solver_batch=rng.choice([8, 16, 32]), **restart, **kinds)
    actions = rng.choice(["continuous", "continuous", "discrete"])
    if what < 0.62:      # one decision per call
        skip = rng.choice([1, 2, 2, 4])
        observe = "rows" if actions == "discrete" else rng.choice(["rows", "fused rows"])
        return _case(dims, _log_int(rng, 16, 131072), skip, frame_skip=skip, actions=actions, observe=observe, **restart, **kinds)
    n_envs = _log_int(rng, 16, 131072)      # fused rollouts
    n_steps = _log_int(rng, 4, 64)
    return _case(dims, n_envs, max(1, min(n_steps, LARGEST // n_envs)), actions=actions, **restart, **kinds)


class _State:
    """A program that steps envs: the handle, the device buffers it hands over, and the actions of its next few calls."""

    def __init__(self, case, seed):
        self.case = case
        self.levels = _levels(case, seed)
        c = case
        self.env = k2d.Env(self.levels, c["n_envs"], auto_reset=c["reset"], max_episode_steps=c["horizon"], seed=seed, frame_skip=c["frame_skip"],
                           solver_batch=c["solver_batch"], max_fused_steps=max(64, c["n_steps"]))
        env, dev = self.env, self.env.device
        gen = torch.Generator(device=dev).manual_seed(seed + 17)
        rows = -(-c["n_steps"] // c["frame_skip"])

        def some(n):
            shape = (n, c["n_envs"], env.n_actions)
            if c["actions"] == "discrete":
                return torch.randint(0, 3, shape, dtype=torch.int32, device=dev, generator=gen)
            return torch.rand(shape, device=dev, generator=gen) * 2 - 1
        self.actions = [some(rows) for _ in range(2)]
        self.reward = torch.empty((c["n_steps"], c["n_envs"]), dtype=torch.float32, device=dev)
        self.done = torch.empty((c["n_steps"], c["n_envs"]), dtype=torch.uint8, device=dev)
        self.view = (torch.empty((c["n_envs"], 125, 125, 4), dtype=torch.uint8, device=dev) if c["observe"] == "pixels"
                     else torch.empty((c["n_envs"], env.obs_floats), dtype=torch.float32, device=dev))
        # the scenes of a run that has been going on for a while
        for _ in range(6):
            env.step(some(-(-16 // c["frame_skip"])), n_steps=16)
        if c["horizon"]:
            st = env.get_state()
            st["step_count"][:] = np.random.Generator(np.random.PCG64(seed)).integers(0, c["horizon"], c["n_envs"])
            env.set_state(st)
        self.calls = 0


def _levels(c, seed):
    dims = scenes.SceneDims(c["polygons"], c["circles"], c["joints"], c["thrusters"])
    return scenes.make_levels(dims, c["levels"], seed, static_prob=c["static"], triangle_prob=c["triangles"], fixed_prob=c["fixed"], limit_prob=c["limited"])


def prepare(case, seed):
    if case["kind"] == "noop":
        return case, _levels(case, seed)
    return _State(case, seed)


def run(state):
    if isinstance(state, tuple):
        case, levels = state
        return k2d.noop_outcomes(levels, case["n_steps"])
    s, env = state, state.env
    actions = s.actions[s.calls & 1]
    s.calls += 1
    if s.case["observe"] == "fused rows":
        return env.step_obs(actions, s.reward, s.done, s.view, n_steps=s.case["n_steps"])
    env.step(actions, s.reward, s.done, n_steps=s.case["n_steps"])
    if s.case["observe"] == "pixels":
        env.render(s.view)
    else:
        env.obs(s.view)
    return s.reward, s.done, s.view


def work(case):
    """Bytes: what is dynamic of the state in and out, actions, reward, done, the observation, and each level's record once.
    Operations: the step as specified, a multiply-add counted as two, with the contacts such scenes have on average."""
    P, C, J, T = case["polygons"], case["circles"], case["joints"], case["thrusters"]
    N, A, E, S = P + C, max(1, J + T), case["n_envs"], case["n_steps"]
    pairs = N * (N - 1) // 2
    manifolds, touching = 0.72 * N, 0.56 * N
    state = 4 * (6 * N + 2 * J + 8 + 5 * touching)
    level = 4 * (12 * N + C + 20 * P + 12 * J + 8 * T + 8)
    flops = (N * 37 + C * 4 + P * 84 + pairs * 8 + J * (107 + 8 * 38) + T * 27 +
             0.7 * P * 190 + 0.8 * C * 94 + touching * 5 + manifolds * (54 + 28 + 8 * 57 + 10))
    moved = case["levels"] * level
    if case["kind"] == "noop":
        moved += E * (state + 1)
    else:
        seen = 62500 if case["observe"] == "pixels" else 4 * (29 * N + 2 * J * (11 + A) + 6 * T)
        moved += E * (2 * state + 4 * A * -(-S // case["frame_skip"]) + 5 * S + seen)
    return {"bytes": moved, "flops": E * S * flops}


def tolerance(case):
    return "exact"
