"""LinGauss actors in BF16 mode: s' = tanh(z + B[a]) + noise, where the scaled normal's product and the addition are rounded once, together."""
import numpy as np
import pytest

from parity_util import blob_for, fields_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,H,N", [(128, 256, 5000), (128, 512, 148 * 128 + 77), (64, 256, 5000), (32, 96, 5000)])
def test_noise_is_added_with_one_rounding(D, H, N):
    """From the zero state z is zero.  A run without noise gives T = tanh(B[a]), one with B = 0 the noise n rounded by itself; T + n rounded
    from these two differs from the fused sum in some rows of every component, and never by more than the last bits of the two."""
    import torch
    from paper_2502_20190_b200 import binding
    A = 5
    rng = np.random.default_rng(D)
    B = rng.uniform(-2, 2, (A, D)).astype(np.float32)
    M = (rng.standard_normal((D, D)) / D).astype(np.float32)

    def next_obs(std, b):
        f = fields_for(env_kind=2, n_envs=N, obs_dim=D, n_actions=A, hidden=H, weight_dtype=1, epsilon=0.3, seed=9, replay_capacity=N * 2,
                       minibatch=16, staleness_bound=2, warmup=0, target_sync_interval=3, gamma=0.99, huber_delta=1.0, lg_done_norm=100.0,
                       lg_noise_std=std, lg_A=M, lg_B=b)
        ctx = binding.Context(**f)
        ctx.publish_weights(blob_for(f, 1))
        ctx.set_state(torch.zeros((N, D), device="cuda"), torch.zeros(N, dtype=torch.int32, device="cuda"))
        ctx.actor_step(1)
        assert ctx.stats()["device_error"] == 0
        return ctx.ring_view()[0][:N, D:2 * D].cpu().numpy()

    T, n, s = next_obs(0.0, B), next_obs(0.01, np.zeros_like(B)), next_obs(0.01, B)
    twice = T + n
    assert np.all(np.abs(s - twice) <= np.spacing(np.abs(twice)) + np.spacing(np.abs(n)))
    # half an ulp of n (2^-31 at 0.01) against an ulp of the sum (2^-24 above a half): some rows in a thousand
    share = np.mean(s != twice, axis=0)
    assert 0 < share.min() and share.max() < 0.2
