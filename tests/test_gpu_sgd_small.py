"""The fused update of small networks where its tiling can go wrong: every row count per block and its edges, several chunks of
rows per block, widths that are no multiple of four (no bulk copies), on both sides of the gradient tile's change, and the largest."""
import pytest

import test_gpu_ppo
import test_gpu_sgd

pytestmark = pytest.mark.gpu
env = test_gpu_sgd.env


@pytest.mark.parametrize("kind,D,A,H,B", [(0, 4, 2, 64, 1), (1, 6, 3, 64, 592), (0, 4, 2, 88, 593), (1, 6, 3, 92, 1185), (0, 4, 2, 128, 2369),
                                          (0, 4, 2, 128, 4737), (1, 6, 3, 20, 8193), (0, 4, 2, 5, 300), (1, 6, 3, 101, 700),
                                          (1, 6, 3, 127, 2400), (2, 8, 4, 40, 77)])
def test_sgd_step(env, kind, D, A, H, B):
    test_gpu_sgd._check_sgd_step(env, kind, D, A, H, 64, B, 0)


@pytest.mark.parametrize("kind,D,A,H,N,T,B", [(1, 6, 3, 101, 40, 10, 257), (0, 4, 2, 128, 300, 10, 2999), (0, 4, 2, 30, 300, 16, 4800)])
def test_ppo_step(env, kind, D, A, H, N, T, B):
    test_gpu_ppo.test_ppo_step_matches_oracle(env, kind, D, A, H, N, T, B, 0)


# hidden 61-64: half of the threads do the narrow gradients beside the hidden matrix's; 8, 16 and 32 rows per block, three outputs and four
@pytest.mark.parametrize("kind,D,A,H,N,T,B", [(0, 4, 2, 64, 100, 10, 1000), (1, 6, 3, 61, 300, 10, 2300), (1, 6, 3, 64, 300, 10, 2999)])
def test_ppo_step_idle_half(env, kind, D, A, H, N, T, B):
    test_gpu_ppo.test_ppo_step_matches_oracle(env, kind, D, A, H, N, T, B, 0)
