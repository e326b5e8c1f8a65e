"""The factor of an ill-conditioned prefix Gram, carried from row to row (no
GPU): the recurrence the team kernel's coefficients come from where the Gram's
pivots would cancel, in numpy float64, held to the backward error of Algorithm 1
(4 n k u, see test_gpu_team_large_vectors); the Gram itself is not.

  H + p p^T, H = L D L^T:  z = L^{-1} p,  Dc as in test_pass_identities,
  D~_q = D_q Dc_q / Dc_{q-1},  L~_iq = L_iq + sigma_q b_q w_iq,
w_iq = p_i - sum_{m<=q} L_im z_m.  And a start from any row's factor L0 D0:
the Grams of L0^{-1} p on top of D0 give L0^{-1} L and the same D."""
from __future__ import annotations

import numpy as np
import pytest

from tests.test_pass_identities import _ldl, _sweep


def _carried(P, sigma, start=None):
    """Per row (a, b, e, Dc) and the factor before the row, carried."""
    n, k = P.shape
    L, D = (np.eye(k), sigma.copy()) if start is None else start
    a, b, e, dc, fac = np.zeros((n, k)), np.zeros((n, k)), np.zeros(n), np.zeros(n), []
    for r in range(n):
        fac.append((L, D))
        w, W = P[r].copy(), np.zeros((k, k))
        for q in range(k):
            w[q + 1:] -= w[q] * L[q + 1:, q]
            W[:, q] = w
        c = 1 + np.cumsum(sigma * w * w / (sigma * D))
        a[r], b[r], e[r], dc[r] = sigma * w, w / (sigma * D * c), c[-1] ** -0.5, c[-1]
        L = L + np.tril(W * (sigma * b[r]), -1)
        D = D * c / np.concatenate([[1.0], c[:-1]])
    return a, b, e, dc, fac


def _gram(P, sigma):
    n, k = P.shape
    a, b, e, dc = np.zeros((n, k)), np.zeros((n, k)), np.zeros(n), np.zeros(n)
    H = np.diag(sigma)
    for r in range(n):
        L, D = _ldl(H)
        z = np.linalg.solve(L, P[r])
        c = 1 + np.cumsum(sigma * z * z / (sigma * D))
        a[r], b[r], e[r], dc[r] = sigma * z, z / (sigma * D * c), abs(c[-1]) ** -0.5, abs(c[-1])
        H = H + np.outer(P[r], P[r])
    return a, b, e, dc


def _backward(F, V, sigma, Lt):
    E = np.longdouble
    A = F.T.astype(E) @ F.astype(E) + (V.astype(E) * sigma) @ V.T.astype(E)
    return float(np.abs(Lt.T.astype(E) @ Lt.astype(E) - A).max() / np.abs(A).max())


@pytest.mark.parametrize("delta,n,k", [(1e-2, 40, 4), (1e-4, 40, 8), (1e-6, 33, 3)])
def test_carried_factor_is_backward_stable_and_the_gram_is_not(delta, n, k):
    rng = np.random.default_rng(n + k)
    F, V, sigma = delta * np.eye(n), rng.standard_normal((n, k)), np.ones(k)
    P = V / delta
    tol = 4 * n * k * 2.0 ** -53
    assert _backward(F, V, sigma, _sweep(F, V, *_carried(P, sigma)[:4])) <= tol
    assert _backward(F, V, sigma, _sweep(F, V, *_gram(P, sigma))) > tol


def test_factor_relative_to_a_start():
    rng = np.random.default_rng(3)
    P, sigma = rng.standard_normal((24, 5)), np.array([1.0, 1, -1, 1, -1])
    P[:, 2] *= 0.1
    P[:, 4] *= 0.05
    fac = _carried(P, sigma)[4]
    L0, D0 = fac[10]
    Y = np.linalg.solve(L0, P[10:20].T).T
    M, D = _ldl(np.diag(D0) + Y.T @ Y)
    np.testing.assert_allclose(L0 @ M, fac[20][0], atol=1e-12)
    np.testing.assert_allclose(D, fac[20][1], rtol=1e-11)
