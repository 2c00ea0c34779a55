"""Evaluation in groups of four and of eight sequence blocks, bit for bit.

Sweeps whose eight-block tasks outnumber the SMs take groups of 256 sequences,
others of 128.  An expert's loss does not depend on the other experts, so many
experts (large groups) agree with one (small groups), at sizes around the
blocks and groups; and the routed path agrees with the oracle elsewhere."""
import numpy as np
import pytest

from gpu_common import run_eval
from paper_2609_37899_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 31, 33, 96, 128, 129, 160, 256, 257, 300, 513])
def test_group_sizes_agree(B):
    E, H, T, N = 16, 66, 4, 40   # 40 experts x (4 + 2) tiles: 240 tasks per group of 256
    theta = inputs.init_params(N, E, H, seed=1)
    bx = inputs.expert_batch(N, B, T, 2, seed=6, step=0)
    many = run_eval(theta, bx, E, H)
    for e in (0, N - 1):
        one = run_eval(theta[e:e + 1], bx[e:e + 1], E, H)
        assert np.array_equal(one, many[e:e + 1])
