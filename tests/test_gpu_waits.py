"""What follows a bounded wait that runs out: the error is reported, outputs are defined, and the device stays usable.

The library is built once more with waits that give up at their first look (TJ_WAIT_POLLS = 0), and each case runs in a process of its
own on that build.  Only kernels whose other waits all end are run this way: the FP32 ones, whose threads go on to the same block
barriers, and the update's TF32 products and the split-operand actor's pairs of blocks, whose issuing warp then issues nothing."""
import os
import subprocess
import sys

import pytest

if __name__ == "__main__":
    sys.path[:0] = [os.path.dirname(os.path.abspath(__file__)), os.path.dirname(os.path.dirname(os.path.abspath(__file__)))]
from parity_util import blob_for, fields_for

pytestmark = pytest.mark.gpu


def _context(kind=0, D=4, A=2, H=64, B=300, N=64, **more):
    import torch
    from paper_2502_20190_b200 import binding
    f = fields_for(env_kind=kind, n_envs=N, obs_dim=D, n_actions=A, hidden=H, epsilon=0.1, seed=5, replay_capacity=N * 8, minibatch=B,
                   staleness_bound=8, warmup=0, target_sync_interval=0, gamma=0.97, huber_delta=1.0)
    f.update(more)
    ctx = binding.Context(**f)
    ctx.publish_weights(blob_for(f, 1))
    return torch, binding, ctx, torch.from_numpy(blob_for(f, 1)).cuda()


def _batch(torch, ctx, n):
    gen = torch.Generator(device="cuda").manual_seed(1)
    b = ctx.alloc_batch(n)
    for k in ("obs", "next_obs", "rew"):
        b[k].normal_(generator=gen)
    b["act"].random_(0, ctx.A, generator=gen)
    b["done"].random_(0, 2, generator=gen)
    return b


def _latched(torch, ctx, code):
    assert ctx.stats()["device_error"] == code
    assert float(torch.ones(1000, device="cuda").sum()) == 1000.0      # the device goes on working


def case_td(H, n, minibatch, kind=0, D=4, A=2):
    torch, binding, ctx, _ = _context(kind, D, A, H, minibatch)
    out = ctx.td_error(_batch(torch, ctx, n))
    _latched(torch, ctx, 3)
    for k in ("td", "huber", "loss"):
        assert bool(torch.isnan(out[k]).all()), k


def case_actor(H, N, steps):
    torch, binding, ctx, _ = _context(H=H, N=N)
    ctx.actor_step(steps)
    ctx.actor_step(steps)
    _latched(torch, ctx, 1)
    assert ctx.stats()["produced"] == 2 * steps * N


def case_split_pairs(kind, D, A, H, N):
    """Neither block of a pair gets its half of the hidden matrix in time: both stop, wait for their copies and leave."""
    torch, binding, ctx, _ = _context(kind, D, A, H, N=N, weight_dtype=2)
    ctx.actor_step(2)
    ctx.actor_step(2)
    _latched(torch, ctx, 4)
    assert ctx.stats()["produced"] == 4 * N


def _unchanged(torch, ctx, blobs, update):
    kept = [b.clone() for b in blobs]
    loss = update()
    _latched(torch, ctx, 3)
    assert bool(torch.isnan(loss).all())
    for a, b in zip(kept, blobs):
        assert torch.equal(a, b)


def case_update(adam, kind, D, A, H, n):
    torch, binding, ctx, theta = _context(kind, D, A, H, n)
    b, target, m, v = _batch(torch, ctx, n), theta.clone(), torch.full_like(theta, 1e-3), torch.full_like(theta, 1e-6)
    if adam:
        _unchanged(torch, ctx, (theta, m, v), lambda: ctx.adam_step(b, 1e-2, theta, target, m, v, 3))
    else:
        _unchanged(torch, ctx, (theta,), lambda: ctx.sgd_step(b, 1e-2, theta, target))


def case_ppo(n):
    torch, binding, ctx, theta = _context(policy_kind=1, epsilon=0.0, replay_capacity=0, rollout_len=8, n_segments=2, B=n)
    x = [torch.rand(n, device="cuda") for _ in range(3)]
    obs, act = torch.randn((n, 4), device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    m, v = torch.full_like(theta, 1e-3), torch.full_like(theta, 1e-6)
    _unchanged(torch, ctx, (theta, m, v), lambda: ctx.ppo_step(obs, act, *x, 1e-2, theta, m, v, 3))


CASES = {
    "td, both networks in shared memory": (case_td, 64, 300, 300),
    "td, both networks in shared memory, several tiles": (case_td, 24, 9000, 300),
    "td, all parameters staged": (case_td, 64, 40, 40, 2, 8, 5),
    "td, all but the hidden matrix staged": (case_td, 256, 70, 8),
    "actor, hidden matrix in shared memory": (case_actor, 64, 1000, 3),
    "actor, two blocks per SM": (case_actor, 64, 6000, 2),
    "actor, hidden matrix through the ring": (case_actor, 256, 500, 3),
    "actor, largest ring": (case_actor, 768, 90, 2),
    "actor, pairs of blocks, split operands": (case_split_pairs, 1, 6, 3, 256, 148 * 128 + 1),
    "actor, pairs of blocks, split operands, two tiles each": (case_split_pairs, 0, 4, 2, 64, 300 * 128),
    "update, fused, SGD": (case_update, False, 0, 4, 2, 64, 300),
    "update, fused, Adam, several chunks of rows per block": (case_update, True, 1, 6, 3, 128, 9000),
    "update, fused, PPO": (case_ppo, 700),
    "update, tensor-core products, SGD": (case_update, False, 2, 32, 7, 512, 3100),
    "update, tensor-core products, Adam": (case_update, True, 2, 32, 7, 512, 3100),
}


@pytest.fixture(scope="module")
def impatient(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_20190_b200 import build
    d = tmp_path_factory.mktemp("impatient")
    return build.compile_library(str(d / "libtj.so"), str(d / "objects"), ["-DTJ_WAIT_POLLS=0"])


@pytest.mark.parametrize("name", list(CASES))
def test_wait_that_runs_out(impatient, name):
    r = subprocess.run([sys.executable, os.path.abspath(__file__), name], env=dict(os.environ, TJ_LIB_PATH=impatient), timeout=120,
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


if __name__ == "__main__":
    fn, *args = CASES[sys.argv[1]]
    fn(*args)
