"""The team kernel (path 1 for factors that stay in L2) at the sizes where its
splits change: orders around its 32-column blocks, its sweep segments (which
start at row blocks 4 s - 2, with other lengths for larger orders and more
vectors) and the three blocks whose tiles the substitution takes apart; vector
counts around its kernels (1, 2, 4, 8) and passes of eight; both signs; padded
and misaligned columns.

Tolerances as in tests/common.py: float64 column-scaled 1e-11 against the
oracle's CholeskyModifyB, float the derived bound against the oracle's mixed
emulation."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_1011_1173_gb300 import chm, inputs
from tests.common import TOL_F64, colscaled_err, tol_mixed

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 0), (32, 2, 0), (33, 1, 3), (64, 8, 1), (96, 9, 0), (97, 4, 2), (128, 1, 0), (129, 17, 0), (160, 2, 4),
          (193, 1, 1), (224, 64, 0), (256, 3, 8), (300, 24, 1), (513, 1, 0), (1100, 5, 0), (2720, 3, 0), (2801, 2, 3)]


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    chm.load(build_if_missing=True)
    torch.cuda.set_device(0)
    chm.config_set("path", chm.PATH_WAVE)
    yield
    chm.config_set("path", chm.PATH_AUTO)


def problem(n, k, pad, dtype):
    L = inputs.spd_factor(n, 300 + n, ld=n + pad).to(dtype)
    L[:, n:] = float("nan")
    V = inputs.update_block(n, k, 300 + n, scale=0.5 / np.sqrt(n * k)).to(dtype)
    return L, V, inputs.sigma_vector(k, 300 + n + k)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n,k,pad", SHAPES)
def test_team_matches_the_oracle(n, k, pad, dtype):
    L, V, sig = problem(n, k, pad, dtype)
    Ld = L.cuda()
    assert chm.modify(Ld, V.cuda(), sig.tolist(), n=n) == chm.CHM_OK
    assert chm.status_sync() == (chm.CHM_OK, -1)
    got = Ld.cpu()
    assert torch.all(torch.isnan(got[:, n:]))
    ref = L[:, :n].contiguous().numpy().copy()
    if dtype == torch.float64:
        assert oracle.modify_b(ref, V.numpy(), sig.numpy())[0] == 0
        tol = TOL_F64
    else:
        assert oracle.modify_mixed32(ref, V.numpy(), sig.numpy(), group=min(k, 64))[0] == 0
        tol = tol_mixed(n, k)
    got = got[:, :n].contiguous().numpy()
    assert colscaled_err(got, ref) <= tol
    low = np.triu(np.ones((n, n), dtype=bool), 1)  # storage row j = column j: above its diagonal lies the lower triangle
    assert np.array_equal(got[low], L[:, :n].numpy()[low])


@pytest.mark.parametrize("k,bad", [(3, 1), (12, 10)])
def test_team_reports_the_row_that_fails(k, bad):
    """A downdate by 2 e_70 of the identity fails at row 70, in the first or a later pass."""
    n = 150
    L = torch.eye(n, dtype=torch.float64, device="cuda")
    V = torch.zeros((k, n), dtype=torch.float64, device="cuda")
    V[bad, 70] = 2.0
    sig = [1] * k
    sig[bad] = -1
    info = torch.full((2,), 9, dtype=torch.int64, device="cuda")
    assert chm.modify(L, V, sig, d_info=info) == chm.CHM_OK
    assert chm.status_sync() == (chm.CHM_ERR_NOT_PD, 70)
    assert info.tolist() == [chm.CHM_ERR_NOT_PD, 70]
