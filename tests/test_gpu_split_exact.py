"""Split-operand kernels (weight mode TJ_W_FP32_TC) on parameters for which every step has one exact value: an identity as the hidden matrix and
inputs, weights and biases of few bits leave nothing to round in front of the head.  What remains -- the split of an activation into two FP16
parts, the order of the head's sums -- is compared bit for bit with its statement in numpy, one tile per SM and pairs of blocks alike."""
import numpy as np
import pytest

from parity_util import fields_for

pytestmark = pytest.mark.gpu

PAIRS = 148 * 128 + 300           # more tiles of 128 envs than SMs


def _fma(w, h, acc):
    """fmaf on values whose exact sum has fewer bits than a double"""
    return (w.astype(np.float64) * h.astype(np.float64) + acc.astype(np.float64)).astype(np.float32)


def _run(kind, on_policy, N, blob, state, W=2):
    import torch
    from paper_2502_20190_b200 import binding
    D, A = ((4, 2), (6, 3))[kind]
    more = dict(policy_kind=1, replay_capacity=0, rollout_len=2, n_segments=2, minibatch=0) if on_policy else dict(
        replay_capacity=N * 4, minibatch=16)
    H = blob["b1"].size
    f = fields_for(env_kind=kind, n_envs=N, obs_dim=D, n_actions=A, hidden=H, weight_dtype=W, epsilon=0.0, seed=3, staleness_bound=2, warmup=0,
                   target_sync_interval=3, gamma=0.99, huber_delta=1.0, **more)
    ctx = binding.Context(**f)
    ctx.publish_weights(np.concatenate([blob[k].ravel() for k in ("W1", "b1", "W2", "b2", "W3", "b3") + (("Wv", "bv") if on_policy else ())]))
    ctx.set_state(torch.from_numpy(state).cuda(), torch.zeros(N, dtype=torch.int32, device="cuda"))
    out = torch.empty((2, N, A), dtype=torch.float32, device="cuda")
    ctx.actor_step(2, out)
    outs = [out[0].cpu().numpy()]
    if on_policy:
        outs.append(ctx.segment_acquire()[1]["val"][0].cpu().numpy()[:, None])
    return np.concatenate(outs, 1), ctx


def _blob(rng, kind, H, on_policy):
    """Hidden unit j sees one input that is a state component; all numbers are multiples of powers of two with few bits."""
    D, A = ((4, 2), (6, 3))[kind]
    b = dict(W1=np.zeros((H, D), np.float32), b1=np.zeros(H, np.float32), W2=np.eye(H, dtype=np.float32))
    first = 0 if kind == 0 else 4                       # Acrobot's inputs 4 and 5 are its angular velocities
    unit_input = first + np.arange(H) % (D - first)
    b["W1"][np.arange(H), unit_input] = rng.choice([-1, 1], H) * 2.0 ** rng.integers(-2, 3, H)
    b["b2"] = (rng.integers(-64, 64, H) / 256).astype(np.float32)
    b["W3"] = (rng.integers(-2047, 2048, (A, H)) / 4096).astype(np.float32)
    b["b3"] = (rng.integers(-64, 64, A) / 256).astype(np.float32)
    if on_policy:
        b["Wv"] = (rng.integers(-2047, 2048, (1, H)) / 4096).astype(np.float32)
        b["bv"] = (rng.integers(-64, 64, 1) / 256).astype(np.float32)
    return b, unit_input


@pytest.mark.parametrize("N", [1, 300, PAIRS])
@pytest.mark.parametrize("kind,H,on_policy", [(0, 64, False), (0, 256, True), (1, 128, False), (1, 192, True), (1, 256, False)])
def test_head_sums_run_over_both_halves_in_column_order(kind, H, on_policy, N):
    rng = np.random.default_rng(H + kind)
    b, unit_input = _blob(rng, kind, H, on_policy)
    state = (rng.integers(-4096, 4096, (N, 4)) / 4096).astype(np.float32)
    got, ctx = _run(kind, on_policy, N, b, state)
    x = state[:, unit_input - 2 if kind else unit_input]                # [N][H]: the input of each unit
    h = np.maximum(np.maximum(b["W1"].sum(1) * x, 0) + b["b2"], 0).astype(np.float32)
    W3, b3 = (np.concatenate([b["W3"], b["Wv"]]), np.concatenate([b["b3"], b["bv"]])) if on_policy else (b["W3"], b["b3"])
    want = np.empty((N, len(b3)), np.float32)
    for a in range(len(b3)):
        half = []
        for c0 in (0, H // 2):
            s = np.zeros(N, np.float32)
            for c in range(c0, c0 + H // 2):
                s = _fma(W3[a, c], h[:, c], s)
            half.append(s)
        want[:, a] = (b3[a] + half[0]) + half[1]
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
    assert ctx.stats()["device_error"] == 0
