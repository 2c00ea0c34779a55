"""The probe sums of the updates, sum_i c_i z_i, element by element: every
probe count around the kernel's groups of four, dense and sparse, and several
accumulation batches.  theta = 0 and lr = n make the SGD update write -G;
beta1 = 0 without decay makes Adam's m the mean of the sums.  n sequential
fp32 additions are off by at most n 2^-24 sum |c| (two more roundings for m)."""
import numpy as np
import pytest
import torch

from gpu_common import api

pytestmark = pytest.mark.gpu

U24 = 2.0 ** -24


def _sums(oracle, P, c, steps, kind):
    G = np.zeros(P)
    for a, st in enumerate(steps):
        for i in range(c.shape[1]):
            G += float(c[a, i]) * oracle.probe(9, st, 0, i, 0, P, kind=kind).astype(np.float64)
    return G


@pytest.mark.parametrize("E,H,n", [(1, 1, 1), (3, 2, 3), (5, 7, 16), (2, 3, 257), (9, 5, 6)])
def test_sgd_sums(oracle_mod, E, H, n):
    P = oracle_mod.param_count(E, H)
    c = np.random.default_rng([E, H, n]).standard_normal((1, n)).astype(np.float32)
    params = torch.zeros(1, P, device="cuda")
    api().spsa_update(params, E, H, float(n), 9, 4, torch.from_numpy(c).cuda())
    err = np.abs(-params.cpu().numpy()[0] - _sums(oracle_mod, P, c, [4], "dense"))
    assert err.max() <= n * U24 * np.abs(c).sum()


@pytest.mark.parametrize("kind", ["sparse", "dense"])
@pytest.mark.parametrize("E,H,n,A", [(1, 1, 1, 1), (3, 2, 15, 1), (5, 7, 40, 3)])
def test_adam_sums(oracle_mod, E, H, n, A, kind):
    P = oracle_mod.param_count(E, H)
    c = np.random.default_rng([E, H, n, A]).standard_normal((A, 1, n)).astype(np.float32)
    steps = [3 + 7 * a for a in range(A)]
    z = [torch.zeros(1, P, device="cuda") for _ in range(3)]
    api().adam_update(*z, E, H, kind, 9, steps, torch.from_numpy(c).cuda(), 1e-3, 0.0, 0.999, 1e-8,
                      0.0, 1)
    G = _sums(oracle_mod, P, c[:, 0], steps, kind)
    err = np.abs(z[1].cpu().numpy()[0] - G / (A * n))
    assert err.max() <= ((A * n + 2) * U24 * np.abs(c).sum()) / (A * n)
