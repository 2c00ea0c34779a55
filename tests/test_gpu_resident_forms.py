"""The resident kernel's two forms give the same bits.

More (expert, probe) pairs than SMs run two CTAs per SM (probe tiles in tensor
memory, accumulators that the gate and the head share); fewer run one CTA per
SM (two operand buffers, two head accumulators, probe tiles in tensor or
shared memory).  A probe's losses do not depend on how many probes there are,
so the first probes of a large call equal a small call's."""
import numpy as np
import pytest

from gpu_common import run_step
from paper_2609_37899_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E,H,B,T", [
    (32, 48, 16, 9),   # shared accumulators, two gate tiles, the second half empty
    (16, 24, 5, 6),    # one gate tile, separate accumulators within half of tensor memory
    (20, 30, 17, 4),   # ragged, three 8-sequence groups
    (8, 64, 3, 5),     # the widest expert
    (32, 64, 16, 4),   # too large for two per SM; probe tiles in shared memory
    (64, 16, 1, 1),    # one sequence of one target
])
def test_forms_agree(E, H, B, T):
    theta = inputs.init_params(1, E, H, seed=2)
    bx = inputs.expert_batch(1, B, T, 2, seed=6, step=0)
    few = run_step(theta, bx, E, H, 3, 1e-3, 0.0, 7, 2)
    many = run_step(theta, bx, E, H, 400, 1e-3, 0.0, 7, 2)
    assert few["status"] == 0 and many["status"] == 0
    assert np.array_equal(few["losses"], many["losses"][:, :3])
    assert np.array_equal(few["coef"], many["coef"][:, :3])
