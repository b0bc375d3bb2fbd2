"""The scan of the fused path at the sizes where its shape changes: one warp per row up to 32 rows, two rows per warp beyond; up to 144
positions it folds the states itself, above them a kernel before it does; CTA counts below, at and above what a lane has in flight."""
import numpy as np
import pytest

from tests.test_gpu_fused import run_and_check


@pytest.mark.gpu
@pytest.mark.parametrize("B,K,D,V", [
    (2, 31, 64, 640), (2, 32, 64, 640), (1, 63, 64, 640), (1, 62, 64, 640), (144 // 2, 1, 64, 640),
    (16, 8, 64, 4096), (29, 4, 64, 4096),      # 144 positions, 145
    (3, 3, 64, 20480), (3, 3, 64, 256), (1, 1, 64, 8)])
def test_scan_after_the_fused_kernel(B, K, D, V):
    run_and_check(B, K, D=D, V=V, W=min(2, K))
    rng = np.random.default_rng(K)
    W = min(3, K)
    state = np.stack([rng.integers(0, W + 1, B), rng.integers(1, K + 1, B), rng.integers(0, V, B)], axis=1).astype(np.int32)
    state[state[:, 0] == 0] = [0, 0, -1]
    state[0] = [1, -1, 0]                      # no state that a step writes
    run_and_check(B, K, D=D, V=V, W=W, theta=0.5, boundary="carry", state=state.tolist())
