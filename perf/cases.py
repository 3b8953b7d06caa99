"""The work a user of this framework has it do, as cases that can be timed: whole passes through the public entry points
(paper_2104_06272_b200.binding), from the tiny reference loop to the largest batch a GPU is given.

A case is a dict of plain values.  `kind` says which program it stands for:

  train   the training loop: iters x (rollout of T steps, A2C update) by run(iters)
  shard   the same iteration as a replica runs it: rollout, grads, apply_grads (the exchange between them is the caller's)
  ppo     one rollout, then `epochs` clipped-surrogate steps on it
  vtrace  one rollout, then `epochs` V-trace steps on it (every epoch after the first is off-policy)
  act     acting alone, by the entry point for callers without a workspace (evaluation, a control loop)
  host    a host-driven loop: parameters and env state in from page-locked memory, one iteration, the results back out,
          the host waits for them

After a device-side pass the learner's state (parameters, last gradient, Adam moments) and the env state are read into
the program's own device tensors, as for a checkpoint or a publication of weights.

The remaining fields are the configuration: B envs of an N x N board, hidden width H, T steps, precision (0 = fp32,
1 = bf16), env_kind (0 = grid, 1 = torus), n_policies (0 = one policy).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2104_06272_b200 import binding as bnd

FIELDS = dict(env_kind=0, n_policies=0, precision=0, iters=1, epochs=1)


def _case(name, kind, B, N, H, T, **more):
    return {"name": name, "kind": kind, "B": B, "N": N, "H": H, "T": T, **FIELDS, **more}


def listed():
    return [
        # The five workloads the framework is quoted on, at their own sizes (workloads.py); tiny's run is 2 iterations.
        _case("tiny", "train", 64, 5, 64, 16, iters=2),
        _case("throughput", "train", 4096, 10, 256, 32),
        _case("memory_bound", "train", 131072, 8, 128, 64),
        _case("large_batch", "train", 65536, 10, 256, 32),
        _case("tensor_core", "train", 16384, 16, 1024, 32, precision=1),
        # Many small independent networks on one GPU (the benchmark's sixth shape).
        _case("many_policies", "train", 65536, 5, 64, 16, n_policies=1024),
        # A middling PPO job: several epochs on one rollout, each after the first with a recomputed forward pass; torus.
        _case("ppo_epochs", "ppo", 2500, 9, 128, 24, env_kind=1, epochs=4),
        # Off-policy learning in bf16 at a width whose weights stay on chip, a board with more than 128 cells.
        _case("vtrace_bf16", "vtrace", 6000, 12, 256, 20, precision=1, epochs=2),
        # A replica's shard at a width that is no power of two, odd batch.
        _case("shard_width_96", "shard", 777, 7, 96, 20),
        # fp32 at a hidden width common in reinforcement learning and above 256.
        _case("fp32_width_512", "train", 3000, 11, 512, 16),
        # Acting in a control loop that may not allocate: a small odd batch.
        _case("act_noalloc", "act", 1013, 10, 256, 12),
        # The end-to-end form of the headline workload: state from the host and back every iteration.
        _case("host_loop", "host", 4096, 10, 256, 32),
    ]


WIDTHS = (32, 64, 96, 128, 192, 256, 384, 512, 768, 1024)  # every hidden width the library takes
VTRACE_WIDTHS = {0: (64, 128, 256), 1: (64, 128, 256, 512, 1024)}  # ... of them with the V-trace objective
MAX_FLOPS, MAX_ACTS, MAX_ROWS = 3.3e12, 1.0e9, 8.0e6  # of the largest listed cases: arithmetic, saved activations, rows


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("train", "train", "train", "train", "many", "shard", "ppo", "vtrace", "act", "host"))
    N, T, env_kind = rng.randint(3, 16), _log(rng, 4, 64), rng.choice((0, 0, 1))
    precision = rng.choice((0, 0, 1))
    # half of the draws at the widths of the framework's own configurations, half anywhere
    H = rng.choice((64, 128, 256) if rng.random() < 0.5 else WIDTHS)
    if kind == "many":
        K, per = _log(rng, 2, 1024), _log(rng, 8, 256)
        B = K * per - rng.randint(0, min(K, per) - 1)
        c = _case("", "train", B, N, rng.choice((64, 64, 128)), min(T, 32), env_kind=env_kind, n_policies=K)
        del c["name"]
        return c
    B, epochs = _log(rng, 32, 131072), 1
    if kind == "vtrace":
        H = rng.choice(VTRACE_WIDTHS[precision])
    if kind in ("ppo", "vtrace"):
        epochs = rng.randint(2, 4)
    if kind == "act":
        precision, T, B = 0, min(T, 32), min(B, 4096, bnd.NOALLOC_MAX_BH // H)
    c = _case("", kind, B, N, H, T, env_kind=env_kind, precision=precision, epochs=epochs)
    del c["name"]
    # no dearer than the largest listed case
    over = max(work(c)["flops"] / MAX_FLOPS, B * T * H / MAX_ACTS, B * T / MAX_ROWS)
    if over > 1:
        c["B"] = max(1, int(B / over))
    return c


def _config(case):
    return bnd.make_cfg(case["B"], case["N"], case["H"], case["T"], precision=case["precision"], env_kind=case["env_kind"],
                        n_policies=case["n_policies"])


def _initial_params(an):
    """The library's own initialisation with the policy head scaled down to a hundredth, as is usual for the last layer
    of a policy: training starts near the uniform policy."""
    theta = an.get(bnd.PARAMS).reshape(an.K, an.P)
    heads = theta[:, an.P - 5 - 5 * an.H: an.P - 5].reshape(an.K, an.H, 5)
    heads[:, :, :4] *= np.float32(0.01)
    return theta.reshape(-1)


CHECKPOINT = (("params", bnd.PARAMS), ("grads", bnd.GRADS), ("adam_m", bnd.ADAM_M), ("adam_v", bnd.ADAM_V),
              ("pos", bnd.ENV_POS), ("tep", bnd.ENV_TEP))
_TORCH = {bnd.ENV_POS: torch.uint8, bnd.ENV_TEP: torch.uint8}


def prepare(case, seed):
    cfg = _config(case)
    an = bnd.Anakin(cfg)
    an.reset(seed)
    an.set(bnd.PARAMS, _initial_params(an))
    if case["kind"] == "act":
        return _prepare_act(case, cfg, an, seed)
    state = {"case": case, "an": an}
    if case["kind"] == "host":
        pin = lambda a: torch.from_numpy(a).pin_memory()  # noqa: E731
        state["in"] = {w: pin(an.get(w)) for w in (bnd.PARAMS, bnd.ENV_POS, bnd.ENV_TEP)}
        state["out"] = {w: pin(an.get(w)) for w in (bnd.PARAMS, bnd.ENV_POS, bnd.ENV_TEP)}
        state["grads"] = pin(an.get(bnd.GRADS))
        return state
    state["out"] = {name: torch.empty(an.blob_bytes(w) // (1 if w in _TORCH else 4), dtype=_TORCH.get(w, torch.float32),
                                      device=an.device) for name, w in CHECKPOINT}
    return state


def _prepare_act(case, cfg, an, seed):
    def dev(which):
        a = an.get(which)
        return torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).cuda()

    T, B = case["T"], case["B"]
    new = lambda n, dtype: torch.empty(n, dtype=dtype, device="cuda")  # noqa: E731
    return {"case": case, "cfg": cfg, "seed": seed, "step": 0,
            "env": [dev(w) for w in (bnd.PARAMS, bnd.ENV_WALLS, bnd.ENV_START, bnd.ENV_GOAL, bnd.ENV_POS, bnd.ENV_TEP)],
            "traj": [new(T * B, torch.uint8), new(T * B, torch.int8), new(T * B, torch.uint8), new(T * B, torch.float32),
                     new((T + 1) * B, torch.float32), new(T * B, torch.float32)]}


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "act":
        rc = bnd.rollout_noalloc(state["cfg"], state["seed"], state["step"], case["T"], *state["env"], *state["traj"])
        if rc != bnd.OK:
            raise bnd.AnakinError(rc)
        state["step"] += case["T"]
        return {"env": state["env"][4:], "traj": state["traj"]}
    an = state["an"]
    if kind == "host":
        for w, t in state["in"].items():
            an.set(w, t)
        an.run(case["iters"])
        for w, t in state["out"].items():
            an.get_into(w, t, wait=False)
        an.get_into(bnd.GRADS, state["grads"], wait=False)
        if an.status() != 0:  # waits for the results; they are the next iteration's input
            raise RuntimeError("device status")
        state["in"], state["out"] = state["out"], state["in"]
        return {"state": list(state["in"].values()), "grads": state["grads"]}
    if kind == "train":
        an.run(case["iters"])
    elif kind == "shard":
        an.rollout()
        an.grads()
        an.apply_grads()
    elif kind == "ppo":
        an.rollout()
        an.learn_ppo(case["epochs"], 0.2)
    else:
        an.rollout()
        an.learn_vtrace(case["epochs"], 1.0, 1.0)
    for name, w in CHECKPOINT:
        an.get_into(w, state["out"][name])
    return state["out"]


def work(case):
    """fp32 products count once, however many tensor-core products they are made of.  The first layer is a sum of weight
    rows (its observation is one-hot), computed once per step; backward it is the same sums transposed."""
    B, T, H, N, K = case["B"], case["T"], case["H"], case["N"], max(1, case["n_policies"])
    C = N * N
    P = 3 * C * H + H + H * H + H + 5 * H + 5
    R = B * T
    rows = R + B  # forward passes of a rollout, the bootstrap one among them
    fwd = 2.0 * H * H + 10.0 * H + H
    env = B * (C / 8 + 4.0)  # walls, start, goal, agent cell, clock
    if case["kind"] == "act":
        return {"bytes": 4.0 * P + env + 2.0 * B + 15.0 * R + 4.0 * B, "flops": rows * fwd}
    steps = case["iters"] * (case["epochs"] if case["kind"] in ("ppo", "vtrace") else 1)
    back = 4.0 * H * H + 20.0 * H + H  # gradients of the layer's input and weights
    replays = case["epochs"] - 1 if case["kind"] in ("ppo", "vtrace") else 0
    flops = case["iters"] * rows * fwd + replays * R * fwd + steps * R * back
    # per update: parameters, gradient and moments read and written; per rollout: the env state and the trajectory
    nbytes = steps * K * P * 28.0 + case["iters"] * (env + 2.0 * B + 15.0 * R) + steps * 15.0 * R
    nbytes += 8.0 * K * P * 3  # the state read out at the end
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Sums of 32-bit products agree to about 1e-6, but a unit within rounding of zero (its gate) and a uniform within
    rounding of a boundary (its action) are decisions: one of them moves a gradient by one row's or one env's share.
    Acting alone has no gradient, and so few samples that no action is expected to differ."""
    if case["precision"] == 1:
        return {"rel": 2e-2, "max": 0.9, "differ": 5e-3}
    if case["kind"] == "act":
        return {"rel": 2e-5, "max": 1e-3, "differ": 1e-3}
    return {"rel": 1e-3, "max": 0.3, "differ": 1e-3}
