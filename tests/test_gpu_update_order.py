"""The updates' sums bit for bit, in the order the kernel documents.

Each element's terms are added one by one in fp32, by groups of four probes; inside
a group parameter p begins with probe (p / 32) % 4 of the group and goes round.
theta = 0 and lr = n make the SGD update write -1 * sum; beta1 = 0, no decay and
a power of two for A n make Adam's m the sum over that power, both exact."""
import numpy as np
import pytest
import torch

from gpu_common import api

pytestmark = pytest.mark.gpu


def _sum(oracle, P, c, steps, kind):
    acc = np.zeros(P, np.float32)
    lane = (np.arange(P) // 32) % 4
    n = c.shape[1]
    for a, st in enumerate(steps):
        z = np.stack([oracle.probe(9, st, 0, i, 0, P, kind=kind) for i in range(n)])
        for i0 in range(0, n, 4):
            for k in range(4):
                i = i0 + (lane + k) % 4
                j = np.minimum(i, n - 1)
                term = c[a, j] * z[j, np.arange(P)].astype(np.float32)
                acc = np.where(i < n, acc + term, acc).astype(np.float32)
    return acc


@pytest.mark.parametrize("E,H,n", [(1, 1, 1), (3, 2, 7), (5, 7, 64), (2, 3, 257)])
def test_sgd(oracle_mod, E, H, n):
    P = oracle_mod.param_count(E, H)
    c = np.random.default_rng([E, H, n]).standard_normal((1, n)).astype(np.float32)
    params = torch.zeros(1, P, device="cuda")
    api().spsa_update(params, E, H, float(n), 9, 4, torch.from_numpy(c).cuda())
    assert np.array_equal(-params.cpu().numpy()[0], _sum(oracle_mod, P, c, [4], "dense"))


@pytest.mark.parametrize("kind", ["sparse", "dense"])
@pytest.mark.parametrize("E,H,n,A", [(3, 2, 16, 1), (5, 7, 32, 4), (2, 3, 2, 8)])
def test_adam(oracle_mod, E, H, n, A, kind):
    P = oracle_mod.param_count(E, H)
    c = np.random.default_rng([E, H, n, A]).standard_normal((A, 1, n)).astype(np.float32)
    steps = [3 + 7 * a for a in range(A)]
    z = [torch.zeros(1, P, device="cuda") for _ in range(3)]
    api().adam_update(*z, E, H, kind, 9, steps, torch.from_numpy(c).cuda(), 1e-3, 0.0, 0.999, 1e-8,
                      0.0, 1)
    want = _sum(oracle_mod, P, c[:, 0], steps, kind) / np.float32(A * n)
    assert np.array_equal(z[1].cpu().numpy()[0], want)
