"""The no-allocation variant where its fixed array splits the vectors over
several launches.  In float each launch rounds the diagonal it carried in double,
so the result agrees with the allocating call's one launch within the bound for
float, not bit for bit; in double the launches hold whole passes and it does."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_1011_1173_gb300 import chm, inputs
from tests.common import colscaled_err, tol_mixed
from tests.test_zz_no_alloc import _call


@pytest.mark.gpu
@pytest.mark.parametrize("n,k", [(2048, 64), (1999, 61)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_split_launches(n, k, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    chm.load(build_if_missing=True)
    torch.cuda.set_device(0)
    L0 = inputs.spd_factor(n, n, ld=n + 2).to("cuda", dtype)
    V = inputs.update_block(n, k, n, scale=0.5 / np.sqrt(n * k)).to("cuda", dtype)
    sig = inputs.sigma_vector(k, n).tolist()
    ref, got = L0.clone(), L0.clone()
    info = torch.full((2,), 99, dtype=torch.int64, device="cuda")
    chm.config_set("path", chm.PATH_WAVE)
    try:
        assert _call(chm.chm_modify_ex, ref, V, sig) == chm.CHM_OK
        assert _call(chm.chm_modify_noalloc, got, V, sig, info) == chm.CHM_OK
        torch.cuda.synchronize()
    finally:
        chm.config_set("path", chm.PATH_AUTO)
    assert info.tolist() == [chm.CHM_OK, -1] and chm.status_sync()[0] == chm.CHM_OK
    if dtype == torch.float64:
        assert torch.equal(got, ref)
    else:
        assert colscaled_err(got.cpu().numpy(), ref.cpu().numpy()) <= tol_mixed(n, k)
