"""Cases by which the speed of the sample production/consumption path is measured.

A case is one iteration of a program that uses the library as its users do: produce samples with the actor, consume them
with the learner, publish parameters.  Four loops occur, all through ``binding.Context``:

  td       actor block, staleness-bounded sample, TD error, publish of parameters made elsewhere  (``bench.py``)
  update   actor block, then a number of (sample, SGD or Adam step, publish)                      (``train_dqn.py``)
  rollout  rollout of one segment, acquire, GAE, publish                                          (``bench.py``, on-policy)
  ppo      rollout, acquire, GAE, normalise, epochs of shuffled minibatch updates, publish        (``train_ppo.py``)

Every pass continues where the last one on the same state ended (environments, ring, versions, parameters), as a training
run does.  Sizes are those of the workloads in ``synth.WORKLOADS``, of the training scripts' defaults and of the tests, and
ragged ones between them.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2502_20190_b200 import binding, synth

ENVS = {"cartpole": (synth.ENV_CARTPOLE, 4, 2), "acrobot": (synth.ENV_ACROBOT, 6, 3)}
WEIGHTS = {"fp32": synth.W_FP32, "bf16": synth.W_BF16, "fp32_tc": synth.W_FP32_TC}
GAMMA, LAMBDA = 0.99, 0.95


def _replay(name, loop, env, envs, hidden, minibatch, **more):
    """A case on the replay ring; the keywords override what most of them share."""
    c = dict(name=name, loop=loop, env=env, envs=envs, obs=0, actions=0, hidden=hidden, weights="fp32", minibatch=minibatch,
             actor_steps=4, ring_calls=16, staleness=8, updates=0, optimizer="", host_blob=False, two_stream=False, done_norm=4.0)
    c.update(more)
    if env in ENVS:
        c["obs"], c["actions"] = ENVS[env][1:]
    return c


def _segments(name, loop, env, envs, hidden, rollout, **more):
    """A case on rollout segments."""
    c = dict(name=name, loop=loop, env=env, envs=envs, obs=ENVS[env][1], actions=ENVS[env][2], hidden=hidden, weights="fp32",
             rollout=rollout, minibatch=0, epochs=0)
    c.update(more)
    return c


def listed():
    return [
        # the smallest workload (cfg1): a few environments stepped by a small network, everything a launch or two long
        _replay("cartpole_64_td", "td", "cartpole", 64, 64, 256, ring_calls=256, staleness=4),
        # train_dqn.py as it stands: one actor step, four Adam updates with a publish each
        _replay("cartpole_1024_adam", "update", "cartpole", 1024, 64, 1024, actor_steps=1, ring_calls=128, updates=4, optimizer="adam"),
        # cfg2: an ordinary amount of environments; the parameters come from pinned host memory, as from another process
        _replay("cartpole_4096_td_host", "td", "cartpole", 4096, 128, 1024, ring_calls=64, host_blob=True),
        # the same workload trained, learner on a second stream (train_dqn.py --two-stream)
        _replay("cartpole_4096_adam_2stream", "update", "cartpole", 4096, 128, 1024, ring_calls=64, updates=1, optimizer="adam",
                two_stream=True),
        # sizes that fit no tile: a user's own environment count, width and minibatch
        _replay("acrobot_3001_sgd_ragged", "update", "acrobot", 3001, 100, 777, ring_calls=20, updates=2, optimizer="sgd"),
        # cfg3 with its hidden layer on the tensor cores at FP32 accuracy
        _replay("acrobot_16384_td_tc", "td", "acrobot", 16384, 256, 4096, weights="fp32_tc", ring_calls=64, staleness=4),
        # cfg3 trained in the reproducible FP32 mode
        _replay("acrobot_16384_sgd_fp32", "update", "acrobot", 16384, 256, 4096, ring_calls=64, staleness=4, updates=1, optimizer="sgd"),
        # train_ppo.py as it stands: short segments, four epochs of eight minibatches
        _segments("cartpole_1024x32_ppo", "ppo", "cartpole", 1024, 64, 32, minibatch=4096, epochs=4),
        # cfg4: long rollouts of many environments, then one reverse scan
        _segments("cartpole_65536x128_rollout_tc", "rollout", "cartpole", 65536, 256, 128, weights="fp32_tc"),
        # a wide state on the tensor cores, neither the largest width nor whole tiles; episodes end by the step limit only
        _replay("lingauss64_10000_td_bf16", "td", "lingauss", 10000, 256, 2048, obs=64, actions=8, weights="bf16", ring_calls=8,
                staleness=16, done_norm=16.0),
        # cfg5's network trained: FP32 master parameters beside the BF16 actor, a ragged number of environments
        _replay("lingauss_20000_sgd_bf16", "update", "lingauss", 20000, 512, 8192, obs=128, actions=16, weights="bf16", ring_calls=16,
                staleness=16, updates=1, optimizer="sgd"),
        # cfg5: the largest workload
        _replay("lingauss_262144_td_bf16", "td", "lingauss", 262144, 512, 8192, obs=128, actions=16, weights="bf16", ring_calls=16,
                staleness=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    family = rng.choice(("td_fp32", "update_fp32", "td_tc", "rollout", "ppo", "td_bf16", "update_bf16", "td_bf16_narrow"))
    env = rng.choice(("cartpole", "acrobot"))
    more = dict(actor_steps=rng.choice((1, 2, 4, 8)), ring_calls=_log_int(rng, 8, 64), staleness=rng.choice((4, 8, 16)))
    train = dict(updates=rng.choice((1, 2, 4)), optimizer=rng.choice(("sgd", "adam")))
    if family == "td_fp32":
        c = _replay("", "td", env, _log_int(rng, 16, 8192), _log_int(rng, 24, 200), _log_int(rng, 32, 4096),
                    host_blob=rng.random() < 0.3, **more)
    elif family == "update_fp32":
        c = _replay("", "update", env, _log_int(rng, 64, 4096), _log_int(rng, 24, 256), _log_int(rng, 64, 4096),
                    two_stream=rng.random() < 0.3, **more, **train)
    elif family == "td_tc":
        c = _replay("", "td", env, _log_int(rng, 256, 65536), rng.choice((64, 128, 192, 256)), _log_int(rng, 256, 8192),
                    weights="fp32_tc", **more)
    elif family == "rollout":
        if rng.random() < 0.6:
            c = _segments("", "rollout", env, _log_int(rng, 256, 65536), rng.choice((64, 128, 192, 256)), _log_int(rng, 16, 128),
                          weights="fp32_tc")
        else:
            c = _segments("", "rollout", env, _log_int(rng, 64, 8192), _log_int(rng, 24, 128), _log_int(rng, 16, 128))
    elif family == "ppo":
        c = _segments("", "ppo", env, _log_int(rng, 64, 4096), _log_int(rng, 32, 256), _log_int(rng, 8, 32), epochs=rng.randint(1, 4))
        c["minibatch"] = min(_log_int(rng, 512, 8192), c["envs"] * c["rollout"])
    elif family == "td_bf16_narrow":
        more["ring_calls"] = 8
        c = _replay("", "td", "lingauss", _log_int(rng, 256, 65536), 32 * rng.randint(1, 16), _log_int(rng, 256, 8192),
                    obs=rng.choice((32, 64, 96)), actions=rng.randint(2, 16), weights="bf16", done_norm=rng.choice((4.0, 16.0)), **more)
    else:
        more["actor_steps"], more["ring_calls"] = rng.choice((1, 2, 4)), 8
        big = family == "td_bf16"
        c = _replay("", "td" if big else "update", "lingauss", _log_int(rng, 512, 262144 if big else 65536), rng.choice((128, 256, 384, 512)),
                    _log_int(rng, 256, 8192), obs=128, actions=rng.randint(2, 16), weights="bf16", done_norm=rng.choice((4.0, 16.0)),
                    **more, **({} if big else train))
    del c["name"]
    return c


def _on_policy(c):
    return c["loop"] in ("rollout", "ppo")


def _mid_run_states(c, gen):
    """Environment states and episode positions as they are in the middle of a run: spread over what the dynamics reach."""
    n = c["envs"]
    uni = lambda *s: torch.rand(*s, generator=gen, device="cuda") * 2 - 1  # noqa: E731
    if c["env"] == "cartpole":
        s = torch.stack([1.5 * uni(n), uni(n), 0.15 * uni(n), uni(n)], 1)
    elif c["env"] == "acrobot":
        s = torch.stack([math.pi * uni(n), math.pi * uni(n), 3 * uni(n), 6 * uni(n)], 1)
    else:
        s = uni(n, c["obs"])
    steps = torch.randint(0, 100, (n,), generator=gen, device="cuda", dtype=torch.int32)
    return s.float().contiguous(), steps


class State:
    """What a training program keeps: the context, its parameters, its batch and output arrays."""


def prepare(case, seed):
    c, s = case, State()
    s.case = c
    kind = synth.ENV_LINGAUSS if c["env"] == "lingauss" else ENVS[c["env"]][0]
    fields = dict(env_kind=kind, n_envs=c["envs"], obs_dim=c["obs"], n_actions=c["actions"], hidden=c["hidden"],
                  weight_dtype=WEIGHTS[c["weights"]], seed=seed, gamma=GAMMA, gae_lambda=LAMBDA, huber_delta=1.0)
    if _on_policy(c):
        fields.update(policy_kind=synth.POLICY_CATEGORICAL, epsilon=0.0, replay_capacity=0, rollout_len=c["rollout"], n_segments=3,
                      staleness_bound=2, minibatch=c["minibatch"])
    else:
        fields.update(policy_kind=synth.POLICY_EPS_GREEDY, epsilon=0.1, minibatch=c["minibatch"], staleness_bound=c["staleness"],
                      replay_capacity=c["envs"] * c["actor_steps"] * c["ring_calls"], warmup=0, target_sync_interval=1000)
        if kind == synth.ENV_LINGAUSS:
            fields["lg_done_norm"] = c["done_norm"]
    s.ctx = ctx = binding.Context(**synth.config_fields(fields))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    vh = _on_policy(c)
    blobs = [torch.from_numpy(synth.policy_blob(seed, v + 1, c["obs"], c["hidden"], c["actions"], vh)) for v in range(2)]
    s.theta, s.theta_target = blobs[0].cuda(), blobs[1].cuda()
    s.blobs = [b.pin_memory() if c.get("host_blob") else b.cuda() for b in blobs]
    s.passes = 0
    if c["loop"] in ("update", "ppo"):
        # moments with some history, as after a thousand steps
        s.m = 1e-3 * torch.randn(s.theta.numel(), generator=gen, device="cuda")
        s.v = 1e-6 * (0.5 + torch.rand(s.theta.numel(), generator=gen, device="cuda"))
        s.t = 1000
    ctx.publish_weights(s.theta)
    state, steps = _mid_run_states(c, gen)
    ctx.set_state(state, steps)
    view = ctx.get_state()
    s.out = {"state": view["state"], "ep_step": view["ep_step"]}
    if _on_policy(c):
        s.adv = torch.empty((c["rollout"], c["envs"]), dtype=torch.float32, device="cuda")
        s.ret = torch.empty_like(s.adv)
        if c["loop"] == "ppo":
            rows, s.minibatches = c["rollout"] * c["envs"], {}
            s.shuffles = 0
            for r0 in range(0, rows, c["minibatch"]):
                n = min(rows - r0, c["minibatch"])
                if n not in s.minibatches:
                    s.minibatches[n] = ctx.alloc_minibatch(n)
        return s
    s.batch = ctx.alloc_batch()
    s.out.update({k: v for k, v in s.batch.items() if k != "c"})
    if c["loop"] == "td":
        dev = dict(dtype=torch.float32, device="cuda")
        s.td = dict(td=torch.empty(c["minibatch"], **dev), huber=torch.empty(c["minibatch"], **dev), loss=torch.empty(1, **dev))
        s.out.update(s.td)
    # the ring holds the last few versions' records; the records of one actor call are `rows` consecutive ones
    ring, _ = ctx.ring_view()
    rows = c["envs"] * c["actor_steps"]
    s.records = [ring[i * rows:(i + 1) * rows] for i in range(c["ring_calls"])]
    for _ in range(4):
        ctx.actor_step(c["actor_steps"])
        ctx.publish_weights(s.theta)
    s.actor_calls = 4
    if c["two_stream"]:
        torch.cuda.synchronize()
        ctx.use_learner_stream(True)
    return s


def run(s):
    c, ctx = s.case, s.ctx
    out = dict(s.out)
    s.passes += 1
    if _on_policy(c):
        ctx.actor_step(c["rollout"])
        _, seg = ctx.segment_acquire()
        ctx.gae(seg["rew"], seg["val"], seg["done"], GAMMA, LAMBDA, s.adv, s.ret)
        if c["loop"] == "ppo":
            ctx.normalize(s.adv, 1e-8, out=s.adv)
            rows = c["rollout"] * c["envs"]
            for _ in range(c["epochs"]):
                s.shuffles += 1
                for r0 in range(0, rows, c["minibatch"]):
                    mb = s.minibatches[min(rows - r0, c["minibatch"])]
                    ctx.segment_minibatch(seg, s.adv, s.ret, s.shuffles, r0, mb)
                    s.t += 1
                    out["stats"] = ctx.ppo_step(mb["obs"], mb["act"], mb["logp_old"], mb["adv"], mb["ret"], 3e-4, s.theta, s.m, s.v, s.t)
            ctx.publish_weights(s.theta)
            out.update(theta=s.theta, m=s.m, v=s.v, **{"mb_" + k: v for k, v in mb.items() if k != "c"})
        else:
            ctx.publish_weights(s.blobs[s.passes % 2])
        out.update(adv=s.adv, ret=s.ret, **{k: seg[k] for k in ("obs", "act", "rew", "done", "logp", "val")})
        return out
    ctx.actor_step(c["actor_steps"])
    out["records"] = s.records[s.actor_calls % c["ring_calls"]]
    s.actor_calls += 1
    if c["loop"] == "td":
        ctx.replay_sample(batch=s.batch)
        ctx.td_error(s.batch, s.td)
        if c["host_blob"]:
            blob = s.blobs[s.passes % 2]
            st, _ = binding.tj_publish_weights(ctx.h, blob.data_ptr(), blob.numel() * 4, 0)
            assert st == 0, binding.tj_last_error(ctx.h)
        else:
            ctx.publish_weights(s.blobs[s.passes % 2])
        return out
    for _ in range(c["updates"]):
        ctx.replay_sample(batch=s.batch)
        if c["optimizer"] == "adam":
            s.t += 1
            out["loss"] = ctx.adam_step(s.batch, 5e-4, s.theta, s.theta_target, s.m, s.v, s.t)
        else:
            out["loss"] = ctx.sgd_step(s.batch, 1e-3, s.theta, s.theta_target)
        ctx.publish_weights(s.theta)
    out["theta"] = s.theta
    if c["optimizer"] == "adam":
        out.update(m=s.m, v=s.v)
    return out


def work(case):
    """What one pass cannot do without: multiply-adds of the networks (and of the linear dynamics), states and parameters
    read and written once, records written, sampled rows read and written, the optimiser's arrays."""
    c = case
    D, H, N = c["obs"], c["hidden"], c["envs"]
    A = c["actions"] + (1 if _on_policy(c) else 0)
    macs, blob = D * H + H * H + H * A, D * H + H + H * H + H + H * A + A
    state = D if c["env"] == "lingauss" else 4
    per_step = 2 * macs + (2 * D * D if c["env"] == "lingauss" else 0)
    backward = 2 * macs + 2 * (H * H + H * A)
    flops, nbytes = 0.0, 0.0
    steps = c["rollout"] if _on_policy(c) else c["actor_steps"]
    flops += per_step * N * steps + (2 * macs * N if _on_policy(c) else 0)
    nbytes += N * (2 * state * 4 + 16) + 4 * blob
    if _on_policy(c):
        rows = steps * N
        nbytes += rows * (4 * D + 17) + 4 * N                     # obs, act, rew, logp, val, done; bootstrap values
        nbytes += rows * 17 + 4 * N                               # GAE: rew, val, done in, adv, ret out
        publishes = 1
        if c["loop"] == "ppo":
            nbytes += rows * 8                                    # normalise
            updates = c["epochs"] * -(-rows // c["minibatch"])
            n = c["epochs"] * rows
            nbytes += n * 2 * (4 * D + 16) + n * (4 * D + 16) + updates * 6 * 4 * blob
            flops += n * (2 * macs + backward)
    else:
        rec, B = 4 * (2 * D + 4), c["minibatch"]
        nbytes += N * steps * rec
        if c["loop"] == "td":
            publishes = 1
            nbytes += B * (2 * rec + 4 + rec + 8) + 2 * 4 * blob
            flops += 4 * macs * B
        else:
            publishes = c["updates"]
            nbytes += c["updates"] * (B * (3 * rec + 4) + 4 * blob * (3 if c["optimizer"] == "sgd" else 7))
            flops += c["updates"] * B * (4 * macs + backward)
    nbytes += publishes * 2 * 4 * blob
    return {"bytes": float(nbytes), "flops": float(flops)}


def tolerance(case):
    """Relative error that another correct implementation at the same precision would show.  BF16 weights and activations:
    1e-2.  FP32 forward passes: 1e-5.  Updates: a gradient is a mean of terms of both signs, so the rounding of its sums
    weighs ten times more on what is left.  Actions follow from a comparison of outputs: a few may fall the other way."""
    if case["weights"] == "bf16":
        return {"rel": 1e-2, "differ": 1e-3}
    return {"rel": 1e-4 if case["loop"] in ("update", "ppo") else 1e-5, "differ": 1e-4}
