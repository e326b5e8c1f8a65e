"""chm_solve's chains: every split of the right-hand sides over chains (one,
two or four per chain, the last chain partly filled, more than one launch)
against the oracle's textbook substitutions.

Tolerance as for every solve: per right-hand side max |x_gpu - x_orc| <=
1e-12 max |x_orc| in float64 on factors of condition about 5 (both sides
carry forward errors of order kappa n u), 1e-6 for float storage (double
arithmetic, one rounding of X)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_1011_1173_gb300 import chm, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,tol", [(torch.float64, 1e-12), (torch.float32, 1e-6)])
@pytest.mark.parametrize("n,pad,nrhs", [(1, 0, 3), (31, 2, 17), (33, 0, 16), (64, 1, 33), (97, 3, 64), (130, 0, 66),
                                        (200, 0, 32)])
def test_solve_chains(n, pad, nrhs, dtype, tol):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    chm.load(build_if_missing=True)
    L = inputs.spd_factor(n, 60 + n, ld=n + pad).to(dtype)
    B = torch.randn(nrhs, n + pad, dtype=dtype, generator=torch.Generator().manual_seed(n))
    ref = B.double().numpy().copy()
    assert oracle.solve(L.double().numpy(), ref, n=n)[0] == 0
    X = B.cuda()
    assert chm.solve(L.cuda(), X, n=n) == chm.CHM_OK
    assert chm.status_sync() == (chm.CHM_OK, -1)
    X = X.cpu()
    assert torch.equal(X[:, n:], B[:, n:])
    err = np.abs(X[:, :n].double().numpy() - ref[:, :n]).max(axis=1)
    assert np.all(err <= tol * np.abs(ref[:, :n]).max(axis=1)), err.max()


def test_solve_float_scales():
    """A float factor's tile sums scale the values by powers of two and split
    them into three floats: right-hand sides near both ends of the type's
    range, one whose rows differ by 2^100, and a zero one, against the oracle
    to the same 1e-6 of each (the solve is linear, so scaling by a power of two
    changes no rounding until the result leaves the normal range)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    chm.load(build_if_missing=True)
    n = 300
    L = inputs.spd_factor(n, 17).float()
    B = torch.randn(5, n, dtype=torch.float32, generator=torch.Generator().manual_seed(5))
    B[0] *= 2.0 ** -100
    B[1] *= 2.0 ** 100
    B[2, : n // 2] *= 2.0 ** -100
    B[3] = 0.0
    ref = B.double().numpy().copy()
    assert oracle.solve(L.double().numpy(), ref)[0] == 0
    X = B.cuda()
    assert chm.solve(L.cuda(), X) == chm.CHM_OK
    assert chm.status_sync() == (chm.CHM_OK, -1)
    err = np.abs(X.cpu().double().numpy() - ref).max(axis=1)
    assert np.all(err <= 1e-6 * np.abs(ref).max(axis=1)), err
