"""TD error with both networks in shared memory: every register tile and row count where its plan changes, several tiles per block,
widths that are no multiple of four, and the largest width that fits."""
import pytest

import test_gpu_parity

pytestmark = pytest.mark.gpu
env = test_gpu_parity.env


@pytest.mark.parametrize("kind,D,A,H,B", [(0, 4, 2, 8, 40), (1, 6, 3, 64, 593), (0, 4, 2, 101, 1185), (1, 6, 3, 128, 2369), (0, 4, 2, 64, 4800),
                                          (0, 4, 2, 24, 8700), (1, 6, 3, 150, 700), (2, 20, 4, 48, 300)])
def test_td_error(env, kind, D, A, H, B):
    test_gpu_parity.test_td_error_parity(env, kind, D, A, H, B)
