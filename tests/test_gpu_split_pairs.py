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
