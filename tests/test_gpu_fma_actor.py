"""The FP32 actor of the small environments at the sizes where its plan changes: every register tile, the hidden matrix in shared
memory, over the activations and through the ring, widths that are no multiple of four, ragged environment counts."""
import pytest

import test_gpu_parity

pytestmark = pytest.mark.gpu
env = test_gpu_parity.env


@pytest.mark.parametrize("kind,D,A,H,N", [(0, 4, 2, 1, 1), (0, 4, 2, 64, 593), (1, 6, 3, 101, 1185), (0, 4, 2, 128, 2369), (1, 6, 3, 150, 4737),
                                          (1, 6, 3, 256, 8300), (0, 4, 2, 768, 300)])
def test_actor_step(env, kind, D, A, H, N):
    test_gpu_parity.test_small_env_lockstep_ragged_shapes(env, kind, D, A, H, N, 24)
