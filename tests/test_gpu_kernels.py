"""Kernels at the sizes where their tiling, splitting or number formats change.
Tolerances: FP64 results 1e-11 of the largest entry (a few thousand roundings
of 1.1e-16, amplified by at most the factor 2 k1 = 158 of the entropy); mixed
ones 1e-4 (B0), as everywhere in the suite."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h(vl):
    handle = vl.Handle(0)
    yield handle
    handle.close()


def _f64(*shape):
    return torch.empty(shape, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("m", [513, 575, 576, 577])
def test_fit_b_beyond_one_cluster(vl, h, prec, m):
    """The blocked factorisation: last blocks of 1, 63, 64 and 1 rows."""
    rng = np.random.default_rng(m)
    n = 2 * m + 7
    L = np.tril(rng.uniform(-0.4, 0.4, (m, m)) * (rng.random((m, m)) < 3.0 / m), -1)
    perm = rng.permutation(m)
    E = np.empty((m, n))
    E[perm] = np.linalg.solve(np.eye(m) - L, rng.laplace(size=(m, n)))
    order = torch.from_numpy(perm.astype(np.int32)).cuda()
    B0 = _f64(m, m)
    vl.vl_fit_b(h, torch.from_numpy(E).cuda(), order, None, prec, B0, None)
    h.sync()
    ref = oracle.fp64.b0_ldl(E, list(perm))
    assert np.abs(B0.cpu().numpy() - ref).max() <= (1e-4 if prec == "mixed" else 1e-10)
