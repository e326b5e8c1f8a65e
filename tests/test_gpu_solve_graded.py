"""Solves with float factors whose columns differ by tens of orders of magnitude
(A -> D A D, F -> F D): the values of a tile then do too, inversely, and no part
of them may get lost in sums of floats.

x = D^{-1} (F^T F)^{-1} c for the right-hand side D c; D x, all of the size of
c, is held to the solves' tolerance for float storage, 1e-6 of its largest
(double arithmetic on well-conditioned F, one rounding of X), against the
oracle's double substitutions on the same float data."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_1011_1173_gb300 import chm, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [1, 5, 40])
@pytest.mark.parametrize("n,lo,hi", [(300, -15, 15), (300, -18, 18), (197, -20, 20), (300, -25, 25), (130, -36, -30),
                                     (130, -34, 2), (200, 30, 34), (160, 0, 0)])
def test_graded_factor(n, lo, hi, nrhs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    chm.load(build_if_missing=True)
    rng = np.random.default_rng(n + nrhs)
    d = 10.0 ** rng.uniform(lo, hi, n)  # in no order: neighbours in a tile differ as much as any
    L = (np.tril(inputs.spd_factor(n, 9 + n).numpy()) * d[:, None]).astype(np.float32)  # storage row j = column j
    d = d.astype(np.float32).astype(np.float64)
    B = (rng.standard_normal((nrhs, n)) * d).astype(np.float32)
    ref = B.astype(np.float64)
    assert oracle.solve(L.astype(np.float64), ref)[0] == 0
    X = torch.from_numpy(B).cuda()
    assert chm.solve(torch.from_numpy(L).cuda(), X) == chm.CHM_OK
    assert chm.status_sync() == (chm.CHM_OK, -1)
    err = np.abs((X.cpu().numpy().astype(np.float64) - ref) * d).max(axis=1)
    assert np.all(err <= 1e-6 * np.abs(ref * d).max(axis=1)), err.max()
