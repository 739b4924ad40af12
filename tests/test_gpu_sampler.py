"""The sampler's draw and gather kernels at the sizes where their tiling can go wrong: every lanes-per-draw variant, ragged
minibatches, rows that allow no 16-byte stores, and a ring whose eligible blocks wrap round its end."""
import numpy as np
import pytest

from parity_util import blob_for, fields_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,D,A", [(0, 4, 2), (1, 6, 3), (2, 8, 3), (2, 28, 4), (2, 32, 4), (2, 128, 16)])
@pytest.mark.parametrize("B,shift", [(1, 0), (33, 0), (257, 1)])
def test_gathered_rows_and_staleness_counts(kind, D, A, B, shift):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_20190_b200 import binding, build
    build.build()
    N, blocks = 21, 7
    f = fields_for(env_kind=kind, n_envs=N, obs_dim=D, n_actions=A, hidden=32, epsilon=0.2, seed=99, replay_capacity=N * blocks,
                   minibatch=B, staleness_bound=3, warmup=0, target_sync_interval=0, gamma=0.99, huber_delta=1.0)
    ctx = binding.Context(**f)
    for v in range(9):                    # blocks 7, 8 sit in slots 0, 1: the eligible ones (5..8) wrap round the ring's end
        ctx.publish_weights(blob_for(f, v + 1))
        ctx.actor_step(1)
    batch = ctx.alloc_batch()
    if shift:                             # rows at an odd word: no 16-byte stores
        for name in ("obs", "next_obs"):
            batch[name] = torch.empty(B * D + shift, dtype=torch.float32, device="cuda")[shift:].view(B, D)
        batch["c"].obs, batch["c"].next_obs = batch["obs"].data_ptr(), batch["next_obs"].data_ptr()
    ctx.replay_sample(batch=batch)
    ring = ctx.ring_view()[0].cpu().numpy()
    idx = batch["idx"].cpu().numpy()
    assert set(idx // N) <= {0, 1, 5, 6}
    rec = ring[idx]
    assert np.array_equal(batch["obs"].cpu().numpy(), rec[:, :D]) and np.array_equal(batch["next_obs"].cpu().numpy(), rec[:, D:2 * D])
    tail = rec[:, 2 * D:].view(np.int32)
    for k, name in ((0, "act"), (2, "done"), (3, "ver")):
        assert np.array_equal(batch[name].cpu().numpy(), tail[:, k]), name
    assert np.array_equal(batch["rew"].cpu().numpy(), rec[:, 2 * D + 1])
    s = ctx.stats()
    hist = np.bincount(9 - tail[:, 3], minlength=33)
    assert list(hist) == list(s["staleness_hist"]) and s["max_sampled_staleness"] == int((9 - tail[:, 3]).max())
