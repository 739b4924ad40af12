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


@pytest.mark.parametrize("N,H", [(5000, 64), (PAIRS, 128)])
def test_small_activations_keep_their_rounding(N, H):
    """Scaled activations around FP16's smallest normal number, 2^-14: the high part is the value cut to 11 bits and rounded to FP16, the low part
    the rounded remainder; an output that takes one unit is the sum of the two."""
    rng = np.random.default_rng(4)
    b, unit_input = _blob(rng, 0, H, False)
    for k in ("b2", "W3", "b3"):
        b[k][:] = 0
    b["W1"] = np.abs(b["W1"])
    b["W3"][0, 0] = b["W3"][1, H - 1] = 1
    state = np.exp2(rng.uniform(-24, -10, (N, 4))).astype(np.float32)
    got, _ = _run(0, False, N, b, state)
    for out, unit in ((0, 0), (1, H - 1)):
        v = np.float32(16) * b["W1"][unit, unit_input[unit]] * state[:, unit_input[unit]]
        cut = (v.view(np.uint32) & np.uint32(0xFFFFE000)).view(np.float32)
        want = (cut.astype(np.float16).astype(np.float32) + (v - cut).astype(np.float16).astype(np.float32)) / np.float32(16)
        assert (v < 2.0 ** -14).mean() > 0.2
        assert np.array_equal(got[:, out].view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("N", [300, PAIRS])
def test_a_nan_before_the_relu_is_zero_behind_it_as_in_the_fp32_mode(N):
    rng = np.random.default_rng(6)
    b, _ = _blob(rng, 0, 64, True)
    b["W1"][5] = np.nan
    b["b1"][40] = np.nan
    state = (rng.integers(-4096, 4096, (N, 4)) / 4096).astype(np.float32)
    (split, ctx), (fp32, _) = _run(0, True, N, b, state), _run(0, True, N, b, state, W=0)
    assert np.isfinite(fp32).all()
    assert np.allclose(split, fp32, rtol=1e-5, atol=1e-5 * float(np.sqrt(np.mean(fp32 ** 2))))
    assert ctx.stats()["device_error"] == 0
