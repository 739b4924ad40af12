"""The layer-by-layer update at the edges of its tiles: heads of up to four outputs (a warp per row) and of more, each tile height of
the hidden layers, narrow gradients whose last 64-neuron block is ragged, and fewer units than outputs; the TD error by the same layers."""
import pytest

import test_gpu_parity
import test_gpu_ppo
import test_gpu_sgd

pytestmark = pytest.mark.gpu
env = test_gpu_sgd.env


@pytest.mark.parametrize("kind,D,A,H,B", [(1, 6, 3, 129, 17), (0, 4, 2, 193, 2400), (1, 6, 3, 320, 4097), (2, 12, 4, 67, 129),
                                          (2, 8, 5, 128, 300), (2, 12, 16, 9, 65), (2, 36, 7, 256, 1500)])
def test_sgd_step(env, kind, D, A, H, B):
    test_gpu_sgd._check_sgd_step(env, kind, D, A, H, 64, B, 0)


@pytest.mark.parametrize("kind,D,A,H,N,T,B", [(1, 6, 3, 129, 40, 10, 257), (0, 4, 2, 256, 300, 10, 2999), (0, 4, 2, 200, 20, 4, 40)])
def test_ppo_step(env, kind, D, A, H, N, T, B):
    test_gpu_ppo.test_ppo_step_matches_oracle(env, kind, D, A, H, N, T, B, 0)


@pytest.mark.parametrize("kind,D,A,H,B", [(1, 6, 3, 161, 33), (0, 4, 2, 256, 4097), (1, 6, 3, 256, 15), (2, 12, 4, 333, 300), (0, 4, 2, 768, 130)])
def test_td_error(env, kind, D, A, H, B):
    test_gpu_parity.test_td_error_parity(env, kind, D, A, H, B)
