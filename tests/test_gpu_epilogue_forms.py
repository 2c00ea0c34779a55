"""The persistent kernel's two epilogue widths give the same bits.

Sweeps with more tasks than SMs and few stages along K run 16 epilogue warps,
others 8.  A probe's losses do not depend on how many probes there are, so the
first probes of a large call equal a small call's (three probes: the last
group of a two-probe layout is half empty there, and full in the large one)."""
import numpy as np
import pytest
import torch

from gpu_common import api
from paper_2609_37899_gb300 import inputs

pytestmark = pytest.mark.gpu


def _estimate(theta, bx, E, H, n, kind):
    a = api()
    N, B, T1 = bx.shape
    ws = a.alloc_workspace(E, H, N, n, B, T1 - 1)
    losses = torch.full((N, n, 2), float("nan"), device="cuda")
    coef = torch.full((N, n), float("nan"), device="cuda")
    a.spsa_estimate(torch.from_numpy(theta).cuda(), torch.from_numpy(bx).cuda(), E, H, n, kind,
                    1e-3, 3, 2, losses, coef, ws)
    assert a.get_status() == 0
    return losses.cpu().numpy(), coef.cpu().numpy()


@pytest.mark.parametrize("kind", ["dense", "sparse"])
@pytest.mark.parametrize("E,H,B,T", [
    (16, 100, 40, 5),   # one probe per group, five 8-sequence chunks
    (32, 70, 8, 9),     # two probes per group, one chunk: warps without a share
    (70, 300, 31, 4),   # seven stages, ragged everywhere
    (16, 66, 64, 3),    # the largest group
    (64, 384, 3, 2),
])
def test_widths_agree(E, H, B, T, kind):
    theta = inputs.init_params(1, E, H, seed=1)
    bx = inputs.expert_batch(1, B, T, 2, seed=6, step=0)
    L1, c1 = _estimate(theta, bx, E, H, 3, kind)
    L2, c2 = _estimate(theta, bx, E, H, 201, kind)
    assert np.array_equal(L1, L2[:, :3]) and np.array_equal(c1, c2[:, :3])
