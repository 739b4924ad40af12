"""TD errors of FP32 networks have one rounding order, whichever kernels a call takes: a batch within the configured minibatch, a larger
one and tj_td_error_static give the same bits, and the Q values are those of the oracle's FMA chain."""
import numpy as np
import pytest

import test_gpu_parity
from parity_util import blob_for, fields_for

pytestmark = pytest.mark.gpu
env = test_gpu_parity.env


def _td(torch, call, batch):
    n = batch["c"].n
    out = [torch.full((m,), 7.0, device="cuda") for m in (n, n, 1)]
    assert call(batch["c"], *[x.data_ptr() for x in out]) == 0
    return [x.cpu().numpy() for x in out]


@pytest.mark.parametrize("kind,D,A,H,B", [(0, 4, 2, 40, 700), (0, 4, 2, 150, 40), (1, 6, 3, 161, 33), (2, 12, 4, 190, 17), (0, 4, 2, 193, 31),
                                          (1, 6, 3, 256, 15), (0, 4, 2, 256, 4097), (2, 12, 4, 333, 300), (0, 4, 2, 768, 130)])
def test_one_rounding_order(env, kind, D, A, H, B):
    torch, orc, binding = env
    f = fields_for(env_kind=kind, n_envs=32, obs_dim=D, n_actions=A, hidden=H, epsilon=0.1, seed=5, replay_capacity=32 * 8, minibatch=B,
                   staleness_bound=4, warmup=0, target_sync_interval=0, gamma=0.97, huber_delta=0.8)
    ctx, narrow = binding.Context(**f), binding.Context(**dict(f, minibatch=max(1, B // 2)))
    blob = blob_for(f, 1)
    blob += 0.05 * np.random.default_rng(2).standard_normal(blob.size).astype(np.float32)       # biases too
    for c in (ctx, narrow):
        c.publish_weights(blob)
    gen = torch.Generator(device="cuda").manual_seed(H)
    batch = ctx.alloc_batch()
    for k in ("obs", "next_obs", "rew"):
        batch[k].normal_(generator=gen)
    batch["act"].random_(0, A, generator=gen)
    batch["done"].random_(0, 2, generator=gen)
    got = [_td(torch, lambda b, *o: binding.tj_td_error(ctx.h, b, *o), batch),
           _td(torch, lambda b, *o: binding.tj_td_error_static(ctx.h, b, *o), batch),
           _td(torch, lambda b, *o: binding.tj_td_error(narrow.h, b, *o), batch)]
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a.view(np.int32), b.view(np.int32))
    # without reward and bootstrap term the TD error is -Q(s, a)
    batch["rew"].zero_()
    batch["done"].fill_(1)
    q = -_td(torch, lambda b, *o: binding.tj_td_error(ctx.h, b, *o), batch)[0]
    obs, act = batch["obs"].cpu().numpy(), batch["act"].cpu().numpy()
    rows = sorted(set(range(min(B, 40))) | {B - 1})
    assert np.array_equal(q[rows], [orc.mlp_forward(blob, D, H, A, obs[j])[act[j]] for j in rows])
    for c in (ctx, narrow):
        assert c.stats()["device_error"] == 0
