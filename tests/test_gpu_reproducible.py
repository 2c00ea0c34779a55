"""The step is a fixed sequence of sums: the same inputs give the same bits.

Shapes whose tasks hold few, short stages on the persistent kernel (small
batches, one or two stages along K) are the ones where a task could be
published before its last epilogue warp had written its part."""
import numpy as np
import pytest

from gpu_common import run_step
from paper_2609_37899_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,E,H,n,B,T", [
    (3, 50, 200, 37, 70, 48),   # two sweeps, the second of six sequences
    (2, 16, 96, 33, 5, 64),     # eight-sequence groups, short stages, an odd probe count
    (1, 32, 70, 64, 17, 64),
])
def test_step_is_reproducible(N, E, H, n, B, T):
    theta = inputs.init_params(N, E, H, seed=3)
    bx = inputs.expert_batch(N, B, T, 2, seed=4, step=0)
    first = run_step(theta, bx, E, H, n, 1e-3, 1e-3, 5, 1)
    assert first["status"] == 0
    for _ in range(4):
        again = run_step(theta, bx, E, H, n, 1e-3, 1e-3, 5, 1)
        for k in ("losses", "coef", "theta"):
            assert np.array_equal(first[k], again[k]), k
