"""The body kernel's two forms give the same bits.

More (expert, probe, chunk) streams than SMs run two per CTA, fewer run one.
A probe's losses do not depend on how many probes there are, so the first
probes of a large call equal a small call's; odd stream counts leave the
last CTA of an expert with one stream."""
import numpy as np
import pytest
import torch

from gpu_common import api
from paper_2609_37899_gb300 import inputs

pytestmark = pytest.mark.gpu


def _losses(theta, head, bx, D, n, kind):
    a = api()
    N, B, T1 = bx.shape
    params = torch.from_numpy(theta).cuda()
    losses = torch.full((N, n, 2), float("nan"), device="cuda")
    coef = torch.full((N, n), float("nan"), device="cuda")
    ws = a.body_alloc_workspace(32, D, N, n, B, T1 - 1)
    a.body_spsa_estimate(params, torch.from_numpy(head).cuda(), torch.from_numpy(bx).cuda(), 32, D,
                         n, kind, 1e-3, 3, 2, losses, coef, ws)
    assert a.get_status() == 0
    return losses.cpu().numpy(), coef.cpu().numpy()


@pytest.mark.parametrize("N,D,B,T,few,many,kind", [
    (2, 2, 16, 7, 3, 101, "sparse"),   # odd stream count, whole chunks
    (1, 1, 37, 5, 2, 75, "dense"),     # three chunks, the last ragged, odd
    (3, 2, 1, 1, 4, 70, "sparse"),     # one sequence of one target
])
def test_forms_agree(N, D, B, T, few, many, kind):
    theta = inputs.init_body(N, 32, D, seed=1)
    head = inputs.init_head(32, seed=2)
    bx = inputs.expert_batch(N, B, T, 2, seed=6, step=0)
    L1, c1 = _losses(theta, head, bx, D, few, kind)
    L2, c2 = _losses(theta, head, bx, D, many, kind)
    assert np.array_equal(L1, L2[:, :few]) and np.array_equal(c1, c2[:, :few])
