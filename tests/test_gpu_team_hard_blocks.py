"""Path 1 on factors whose diagonal blocks are ill-conditioned (smooth rows over
a small diagonal), with vectors F^T q, whose substitution is as small as q: a
block's inverse times a residual is off by that block's condition, so such
blocks have to be substituted row by row.

The factor's error against the exact modified factor (Cholesky in extended
precision of the same float64 or float32 data), column-scaled, may be four
times the serial oracle's plus 64 roundings: both are what a stable method
leaves, a few roundings times the conditioning of the factor itself (a
block's inverse instead costs one to two orders of magnitude from a diagonal of
1e-4 on, in float from about 1e-13, which float data does not reach)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_1011_1173_gb300 import chm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    chm.load(build_if_missing=True)
    torch.cuda.set_device(0)
    chm.config_set("path", chm.PATH_WAVE)
    yield
    chm.config_set("path", chm.PATH_AUTO)


def exact_factor(A):
    """The lower factor of A in A's own (extended) precision."""
    A = A.copy()
    L = np.zeros_like(A)
    for j in range(A.shape[0]):
        L[j:, j] = A[j:, j] / np.sqrt(A[j, j])
        A[j + 1:, j + 1:] -= np.outer(L[j + 1:, j], L[j + 1:, j])
    return L


def error(got, exact):
    return float((np.abs(np.tril(got) - exact) / np.abs(exact).max(axis=1, keepdims=True)).max())


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n,k,width,nugget", [(160, 1, 0.002, 1e-4), (161, 4, 0.002, 1e-6), (130, 1, 0.02, 1e-8),
                                              (96, 8, 0.02, 1e-10), (200, 12, 0.002, 1e-8), (33, 2, 0.2, 1e-6),
                                              (150, 3, 0.02, 1e-2)])
def test_factor_error(n, k, width, nugget, dtype):
    f32 = dtype == torch.float32
    if f32:
        nugget = max(nugget, 1e-4)
    rng = np.random.default_rng(n + k)
    x = np.sort(rng.uniform(0, 1, n))
    L = np.linalg.cholesky(np.exp(-np.subtract.outer(x, x) ** 2 / width) + nugget * np.eye(n))
    V = 0.3 * rng.standard_normal((k, n)) @ L.T
    storage = np.float32 if f32 else np.float64
    L, V, sig = L.astype(storage), V.astype(storage), np.ones(k, dtype=np.int8)
    E = np.longdouble
    exact = exact_factor(L.astype(E) @ L.T.astype(E) + V.T.astype(E) @ V.astype(E))
    ref = L.copy()
    assert (oracle.modify_mixed32(ref, V, sig, group=min(k, 64)) if f32 else oracle.modify_b(ref, V, sig))[0] == 0
    Ld = torch.from_numpy(L.copy()).cuda()
    assert chm.modify(Ld, torch.from_numpy(V).cuda(), sig.tolist()) == chm.CHM_OK
    assert chm.status_sync() == (chm.CHM_OK, -1)
    err, tol = error(Ld.cpu().numpy(), exact), 4 * error(ref, exact) + 64 * (2.0 ** -24 if f32 else 2.0 ** -53)
    assert err <= tol, (err, tol)
