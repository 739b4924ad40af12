"""Two contexts of different sizes driven from two host threads: what a kernel's launches share on the device (the limit of its shared
memory) must not depend on which of them set it last.  No launch is refused, and each context ends as it does alone, bit for bit."""
import threading

import pytest

import test_gpu_two_stream
from parity_util import blob_for, fields_for

pytestmark = pytest.mark.gpu
env = test_gpu_two_stream.env
CALLS = 400


def _loop(torch, binding, H, wd, out, start=None):
    try:
        with torch.cuda.stream(torch.cuda.Stream()):
            f = fields_for(env_kind=0, n_envs=64, obs_dim=4, n_actions=2, hidden=H, epsilon=0.1, seed=33, weight_dtype=wd,
                           replay_capacity=64 * 8, minibatch=64, staleness_bound=8, warmup=0, target_sync_interval=3, gamma=0.99, huber_delta=1.0)
            ctx = binding.Context(**f)
            theta = torch.from_numpy(blob_for(f, 1)).cuda()
            target = theta.clone()
            ctx.publish_weights(theta)
            ctx.actor_step(2)
            batch = ctx.alloc_batch()
            if start is not None:
                start.wait(60)
            for _ in range(CALLS):
                ctx.actor_step(1)
                ctx.replay_sample(batch=batch)
                td = ctx.td_error(batch)
                ctx.sgd_step(batch, 1e-3, theta, target)
                ctx.publish_weights(theta)
            assert ctx.wait(0, 60000) == 0
            out[H] = (theta.cpu(), td["td"].cpu(), ctx.ring_view()[0].view(torch.int32).cpu(), ctx.stats()["device_error"])
    except BaseException as e:      # reported by the test's own thread
        out[H] = e


@pytest.mark.parametrize("wd,widths", [(0, (112, 128)), (0, (256, 224)), (2, (64, 256))])
def test_two_contexts_on_two_threads(env, wd, widths):
    torch, binding = env
    alone, together = {}, {}
    for H in widths:
        _loop(torch, binding, H, wd, alone)
    start = threading.Barrier(2)
    threads = [threading.Thread(target=_loop, args=(torch, binding, H, wd, together, start)) for H in widths]
    for t in threads:
        t.start()
    for t in threads:
        t.join(240)
    for H in widths:
        for got in (alone[H], together[H]):
            if isinstance(got, BaseException):
                raise got
        assert together[H][3] == 0
        for a, b in zip(alone[H][:3], together[H][:3]):
            assert torch.equal(a, b), H
