"""Several steps in one launch of the tensor-core actors (128 state components: pipelined; others: serial) against one launch per step: a block with one tile, blocks with one and two, blocks
with several, a ring that wraps inside the call and one that a call writes more than once.  Bit for bit."""
import numpy as np
import pytest

import test_gpu_two_stream
from parity_util import blob_for, fields_for

pytestmark = pytest.mark.gpu
env = test_gpu_two_stream.env


@pytest.mark.parametrize("D,H,N,blocks,calls", [(128, 128, 1, 5, (3, 4)), (128, 512, 100, 4, (2, 7)), (128, 128, 128 * 150 + 5, 6, (5, 4)),
                                                (128, 256, 128 * 400, 3, (2, 3)), (32, 64, 1, 5, (3, 4)), (64, 512, 200, 4, (2, 7)),
                                                (64, 128, 128 * 150 + 5, 6, (5, 4)), (96, 96, 128 * 400, 3, (2, 3))])
def test_steps_of_a_call_equal_single_steps(env, D, H, N, blocks, calls):
    torch, binding = env
    f = fields_for(env_kind=2, n_envs=N, obs_dim=D, n_actions=7, hidden=H, epsilon=0.2, seed=91, weight_dtype=1, replay_capacity=N * blocks,
                   minibatch=1, staleness_bound=4, warmup=0, target_sync_interval=5, gamma=0.99, huber_delta=1.0, max_episode_steps=3,
                   lg_done_norm=9.0)
    got = []
    for single in (False, True):
        ctx = binding.Context(**f)
        for i, n in enumerate(calls):
            ctx.publish_weights(torch.from_numpy(blob_for(f, i + 1)).cuda())
            for _ in range(n if single else 1):
                ctx.actor_step(1 if single else n)
        ring, ver = ctx.ring_view()
        view, s = ctx.get_state(), ctx.stats()
        got.append([a.view(torch.int32).cpu().numpy().copy() for a in (ring, ver, view["state"], view["ep_step"])] +
                   [np.int64([s["episodes_finished"], s["produced"], s["device_error"]])])
    assert got[0][-1][2] == 0 and got[0][-1][0] > 0
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("D,H,N", [(128, 256, 100), (128, 128, 128 * 150 + 5), (32, 64, 300), (64, 128, 128 * 150 + 5)])
def test_network_outputs_and_returns_of_every_step(env, D, H, N):
    """The outputs of step i lie at [i][N][A] and nowhere else; an episode's return is summed from step to step inside the launch."""
    torch, binding = env
    A, steps = 7, 5
    f = fields_for(env_kind=2, n_envs=N, obs_dim=D, n_actions=A, hidden=H, epsilon=0.2, seed=92, weight_dtype=1, replay_capacity=N * 6,
                   minibatch=1, staleness_bound=4, warmup=0, target_sync_interval=5, gamma=0.99, huber_delta=1.0, max_episode_steps=3,
                   lg_done_norm=9.0)
    got = []
    for single in (False, True):
        ctx = binding.Context(**f)
        ctx.publish_weights(torch.from_numpy(blob_for(f, 1)).cuda())
        out = torch.full((steps * N * A + 1024,), -77.0, device="cuda")
        if single:
            for i in range(steps):
                ctx.actor_step(1, out[i * N * A:])
        else:
            ctx.actor_step(steps, out)
        s = ctx.stats()
        assert s["device_error"] == 0 and s["episodes_finished"] >= N
        got.append((out.cpu().numpy(), s["return_sum"]))
    (a, sa), (b, sb) = got
    assert np.all(a[steps * N * A:] == -77.0) and not np.any(a[:steps * N * A] == -77.0)
    assert np.array_equal(a.view(np.int32), b.view(np.int32))
    # the same terms, all negative, in double by atomics in any order: each of the at most steps x N additions of either sum rounds by
    # 2^-53 of the whole at most
    assert abs(sa - sb) <= steps * N * 2.0 ** -52 * abs(sb)
