"""The persistent kernel's two epilogue widths around the lines of their rule.

Sixteen warps run sweeps of more than two 8-sequence chunks per task, up to a number
of stages that depends on the chunks and the probe kind.  A probe's losses do not
depend on how many probes there are, so the first probes of a large call (more
tasks than SMs) equal a small call's (8 warps)."""
import numpy as np
import pytest

from gpu_common import api
from paper_2609_37899_gb300 import inputs
from test_gpu_epilogue_forms import _estimate

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["dense", "sparse"])
@pytest.mark.parametrize("E,H,B,T", [
    (16, 66, 9, 5),     # two probes of two chunks, three stages
    (16, 190, 16, 4),   # four stages, the last line of sparse probes
    (64, 250, 14, 4),   # five, of dense ones
    (16, 100, 24, 4),   # six chunks
    (40, 310, 27, 3),   # eight chunks, six stages, the last line of sparse probes
])
def test_widths_agree(E, H, B, T, kind):
    few, many = 3, 201
    a = api()
    width = [a.lib().soma_debug_epilogue_warps(a.dims(E, H), 1, n, a.PROBE_KINDS[kind], B, 152)
             for n in (few, many)]
    if E != 64 or kind == "dense":
        assert width == [8, 16]
    theta = inputs.init_params(1, E, H, seed=1)
    bx = inputs.expert_batch(1, B, T, 2, seed=6, step=0)
    L1, c1 = _estimate(theta, bx, E, H, few, kind)
    L2, c2 = _estimate(theta, bx, E, H, many, kind)
    assert np.array_equal(L1, L2[:, :few]) and np.array_equal(c1, c2[:, :few])
