"""The resident kernel's two forms under sparse probes and per-probe batches, and
the shapes that only one form takes against the oracle.

More (expert, probe) pairs than SMs run two CTAs per SM, fewer one; a probe's
losses do not depend on how many probes there are, so the first probes of a large
call equal a small call's."""
import numpy as np
import pytest
import torch

from gpu_common import api, assert_coefs, assert_losses, run_step
from paper_2609_37899_gb300 import inputs

pytestmark = pytest.mark.gpu


def _estimate(theta, bx, E, H, n, kind, per_probe):
    a = api()
    N, B, T1 = bx.shape[0], bx.shape[-2], bx.shape[-1]
    losses = torch.full((N, n, 2), float("nan"), device="cuda")
    coef = torch.full((N, n), float("nan"), device="cuda")
    a.spsa_estimate(torch.from_numpy(theta).cuda(),
                    torch.from_numpy(np.ascontiguousarray(bx)).cuda(), E, H, n, kind, 1e-3, 3, 2,
                    losses, coef, a.alloc_workspace(E, H, N, n, B, T1 - 1),
                    batch_per_probe=per_probe)
    assert a.get_status() == 0
    return losses.cpu().numpy(), coef.cpu().numpy()


@pytest.mark.parametrize("kind,per_probe", [("sparse", False), ("dense", True), ("sparse", True)])
@pytest.mark.parametrize("E,H,B,T", [
    (32, 48, 16, 7),   # shared accumulators
    (16, 24, 5, 6),    # separate accumulators
    (20, 30, 17, 4),   # ragged, three 8-sequence groups
])
def test_forms_agree(E, H, B, T, kind, per_probe):
    few, many = 3, 160
    theta = inputs.init_params(1, E, H, seed=2)
    shape = (1, many, B, T + 1) if per_probe else (1, B, T + 1)
    bx = np.random.default_rng([E, H]).integers(0, 256, shape, dtype=np.uint8)
    L1, c1 = _estimate(theta, bx[:, :few] if per_probe else bx, E, H, few, kind, per_probe)
    L2, c2 = _estimate(theta, bx, E, H, many, kind, per_probe)
    assert np.array_equal(L1, L2[:, :few]) and np.array_equal(c1, c2[:, :few])


@pytest.mark.parametrize("E,H,B,T,n", [
    (32, 64, 16, 5, 5),    # probe tiles in shared memory, one CTA per SM
    (32, 64, 16, 5, 155),  # too large for two per SM: the same form with more pairs than SMs
    (32, 48, 16, 5, 155),  # two per SM
])
def test_against_the_oracle(oracle_mod, E, H, B, T, n):
    theta = inputs.init_params(1, E, H, seed=5)
    bx = inputs.expert_batch(1, B, T, 2, seed=8, step=0)
    got = run_step(theta, bx, E, H, n, 1e-3, 1e-2, 4, 1)
    assert got["status"] == 0
    L, c, _ = oracle_mod.spsa_step(theta, E, H, n, np.float32(1e-3), np.float32(1e-2), 4, 1, bx)
    assert_losses(got["losses"], L)
    assert_coefs(got["coef"], c)
