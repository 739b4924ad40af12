"""Publishes from host memory: page-locked blobs that the publish kernel reads itself (up to 512 KB), at an odd offset and up to the last byte of
their allocation, a larger one, and pageable memory, against the same blob on the device."""
import numpy as np
import pytest

from parity_util import blob_for, fields_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,D,A,H,wd", [(0, 4, 2, 61, 0), (1, 6, 3, 128, 0), (0, 4, 2, 256, 2), (2, 64, 8, 256, 1), (2, 128, 16, 512, 1)])
def test_same_outputs_from_every_memory(kind, D, A, H, wd):
    import torch
    from paper_2502_20190_b200 import binding
    N = 200
    f = fields_for(env_kind=kind, n_envs=N, obs_dim=D, n_actions=A, hidden=H, weight_dtype=wd, epsilon=0.1, seed=3, replay_capacity=N * 8,
                   minibatch=64, staleness_bound=8, warmup=0, target_sync_interval=1000, gamma=0.99, huber_delta=1.0)
    blob = torch.from_numpy(blob_for(f, 5))
    n = blob.numel()
    pinned = torch.empty(n + 1, dtype=torch.float32).pin_memory()
    pinned[1:] = blob
    whole = blob.clone().pin_memory()
    outs = []
    for b, on_device in ((blob.cuda(), 1), (whole, 0), (pinned[1:], 0), (blob, 0)):
        ctx = binding.Context(**f)
        assert binding.tj_publish_weights(ctx.h, b.data_ptr(), n * 4, on_device)[0] == 0
        out = torch.empty((N, A), dtype=torch.float32, device="cuda")
        ctx.actor_step(1, out)
        torch.cuda.synchronize()
        outs.append(out.cpu().numpy().view(np.uint32))
    assert all(np.array_equal(outs[0], o) for o in outs[1:])


def test_the_kernel_reads_what_the_memory_holds_when_it_runs():
    """Publishes of one page-locked buffer, rewritten between them once the stream has drained."""
    import torch
    from paper_2502_20190_b200 import binding
    N = 64
    f = fields_for(env_kind=0, n_envs=N, obs_dim=4, n_actions=2, hidden=64, weight_dtype=0, epsilon=0.0, seed=4, replay_capacity=N * 8, minibatch=16,
                   staleness_bound=8, warmup=0, target_sync_interval=1000, gamma=0.99, huber_delta=1.0)
    a, b = binding.Context(**f), binding.Context(**f)
    buf = torch.from_numpy(blob_for(f, 1)).pin_memory()
    for v in range(1, 5):
        buf.copy_(torch.from_numpy(blob_for(f, v)))
        assert binding.tj_publish_weights(a.h, buf.data_ptr(), buf.numel() * 4, 0)[0] == 0
        b.publish_weights(buf.cuda())
        oa, ob = (torch.empty((N, 2), dtype=torch.float32, device="cuda") for _ in range(2))
        a.actor_step(1, oa)
        b.actor_step(1, ob)
        torch.cuda.synchronize()
        assert torch.equal(oa.view(torch.int32), ob.view(torch.int32))
