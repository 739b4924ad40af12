"""Pairs of thread blocks that share the hidden layer's products (weight mode TJ_W_FP32_TC, more tiles of 128 envs than SMs): every width, a
last tile with one env, one whose second block has none, and one that fills both."""
import pytest

from parity_util import RTOL_FP32, blob_for, fields_for

pytestmark = pytest.mark.gpu


def _segment(f, N, T, state, ep):
    import torch
    from paper_2502_20190_b200 import binding
    ctx = binding.Context(**dict(f, n_envs=N))
    ctx.publish_weights(blob_for(f, 1))
    ctx.set_state(state, ep)
    ctx.actor_step(T)
    seg = ctx.segment_acquire()[1]
    return [seg[k].view(torch.uint8).clone() for k in ("obs", "act", "rew", "done", "logp", "val")], ctx


@pytest.mark.parametrize("kind,D,A,H,tiles", [(0, 4, 2, 256, 301), (1, 6, 3, 192, 150)])
def test_a_call_repeats_itself(kind, D, A, H, tiles):
    """64 rollouts from the same states give the same segment bit for bit.  (What a block of a pair hands to the other -- operands in its shared
    memory, accumulators it has read -- is ordered by release and acquire at cluster scope; this would show only a gross lack of it.)"""
    import torch
    N, T = tiles * 128 - 5, 8
    f = fields_for(env_kind=kind, n_envs=N, obs_dim=D, n_actions=A, hidden=H, policy_kind=1, weight_dtype=2, seed=7, replay_capacity=0, rollout_len=T,
                   n_segments=2, staleness_bound=4, gamma=0.99, gae_lambda=0.95, max_episode_steps=5)
    gen = torch.Generator(device="cuda").manual_seed(2)
    state = torch.rand((N, 4), generator=gen, device="cuda") - 0.5
    ep = torch.zeros(N, dtype=torch.int32, device="cuda")
    first, ctx = _segment(f, N, T, state, ep)
    assert ctx.stats()["device_error"] == 0
    for _ in range(63):
        again, _ = _segment(f, N, T, state, ep)
        assert all(torch.equal(a, b) for a, b in zip(first, again))


@pytest.mark.parametrize("kind,D,A,H,tiles,more", [(0, 4, 2, 64, 148, 1), (1, 6, 3, 128, 149, 0), (0, 4, 2, 192, 150, 0), (1, 6, 3, 256, 298, 1)])
def test_outputs_of_every_env_and_step(kind, D, A, H, tiles, more):
    import torch
    from paper_2502_20190_b200 import binding
    N = tiles * 128 + more
    f = fields_for(env_kind=kind, n_envs=N, obs_dim=D, n_actions=A, hidden=H, epsilon=0.2, seed=11, replay_capacity=N * 4, minibatch=19,
                   staleness_bound=2, warmup=N, target_sync_interval=3, gamma=0.99, huber_delta=1.0, max_episode_steps=2)
    many, single, exact = (binding.Context(**dict(f, weight_dtype=w)) for w in (2, 2, 0))
    for c in (many, single, exact):
        c.publish_weights(blob_for(f, 1))
    out = torch.empty((3, N, A), dtype=torch.float32, device="cuda")
    many.actor_step(3, out)
    for t in range(3):
        one, ref = (torch.empty((N, A), dtype=torch.float32, device="cuda") for _ in range(2))
        st = single.get_state()
        exact.set_state(st["state"].clone(), st["ep_step"].clone(), st["cursor"], st["t"], st["k"])
        single.actor_step(1, one)
        exact.actor_step(1, ref)
        assert torch.equal(out[t].view(torch.int32), one.view(torch.int32))          # steps of one launch, launches of one step
        # FP32 sums of the same products in another order, unsplit
        assert torch.all((one - ref).abs() <= RTOL_FP32 * (ref.abs() + ref.pow(2).mean().sqrt()))
    a, b = many.get_state(), single.get_state()
    assert torch.equal(a["state"], b["state"]) and torch.equal(a["ep_step"], b["ep_step"])
    assert many.stats()["device_error"] == single.stats()["device_error"] == 0
    assert many.stats()["episodes_finished"] == single.stats()["episodes_finished"] > 0


@pytest.mark.parametrize("H", [64, 256])
def test_segments_of_every_env_and_step(H):
    """On-policy pairs: outputs and values of every environment, step and bootstrap state equal bit for bit what one tile per SM computes from
    the same states; log-probabilities, rewards, done flags and transitions follow from them."""
    import torch
    from paper_2502_20190_b200 import binding
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N, N0, T = (2 * sms + 3) * 128 + 1, sms * 128, 6
    f = fields_for(env_kind=0, n_envs=N, obs_dim=4, n_actions=2, hidden=H, policy_kind=1, weight_dtype=2, seed=8, replay_capacity=0, rollout_len=T,
                   n_segments=2, staleness_bound=4, gamma=0.99, gae_lambda=0.95, max_episode_steps=4)
    many, few = binding.Context(**f), binding.Context(**dict(f, n_envs=N0, rollout_len=1))
    many.publish_weights(blob_for(f, 1))
    few.publish_weights(blob_for(f, 1))
    gen = torch.Generator(device="cuda").manual_seed(3)
    many.set_state(torch.rand((N, 4), generator=gen, device="cuda") - 0.5, torch.zeros(N, dtype=torch.int32, device="cuda"))
    out = torch.empty((T, N, 2), dtype=torch.float32, device="cuda")
    many.actor_step(T, out)
    seg = {k: v.clone() for k, v in many.segment_acquire()[1].items() if torch.is_tensor(v)}
    states = torch.cat([seg["obs"], many.get_state()["state"][None]])
    one = torch.empty((N0, 2), dtype=torch.float32, device="cuda")
    for t in range(T + 1):
        for c in range(0, N, N0):
            n = min(N0, N - c)
            s = torch.zeros((N0, 4), device="cuda")
            s[:n] = states[t, c:c + n]
            few.set_state(s, torch.zeros(N0, dtype=torch.int32, device="cuda"), t=few.get_state()["t"])
            few.actor_step(1, one)
            val = few.segment_acquire()[1]["val"][0]
            assert torch.equal(val[:n].view(torch.int32), seg["val"][t, c:c + n].view(torch.int32))
            if t < T:
                assert torch.equal(one[:n].view(torch.int32), out[t, c:c + n].view(torch.int32))
    logp = torch.log_softmax(out.double(), -1).gather(-1, seg["act"].long()[..., None])[..., 0]
    assert (logp - seg["logp"]).abs().max() < 1e-5 * (1 + logp.abs().max())
    assert torch.all(seg["rew"] == 1)
    x, v, th, w = seg["obs"].double().unbind(-1)
    force = 20.0 * seg["act"].double() - 10.0
    tmp = (force + 0.05 * w * w * th.sin()) / 1.1
    acc = (9.8 * th.sin() - th.cos() * tmp) / (0.5 * (4.0 / 3.0 - 0.1 * th.cos() ** 2 / 1.1))
    after = torch.stack([x + 0.02 * v, v + 0.02 * (tmp - 0.05 * acc * th.cos() / 1.1), th + 0.02 * w, w + 0.02 * acc], -1)
    done = seg["done"].bool()
    beyond = (after[..., 0].abs() > 2.4) | (after[..., 2].abs() > 12 * 3.14159265358979 / 180)
    near = ((after[..., 0].abs() - 2.4).abs() < 1e-5) | ((after[..., 2].abs() - 12 * 3.14159265358979 / 180).abs() < 1e-5)
    episode = torch.zeros(N, dtype=torch.int32, device="cuda")
    for t in range(T):
        episode += 1
        assert torch.all((done[t] == (beyond[t] | (episode >= 4))) | near[t])
        episode[done[t]] = 0
        assert torch.all(((after[t] - states[t + 1]).abs().amax(-1) < 1e-5) | done[t])
        assert torch.all(states[t + 1][done[t]].abs() <= 0.05)
    assert done.any() and not done.all()
