"""A stream that has solved once holds the workspace of every smaller solve:
no allocation (and so no synchronisation, which a stream capture would not
survive) on a later call of the same or a smaller order with as many
right-hand sides."""
from __future__ import annotations

import pytest
import torch

from paper_1011_1173_gb300 import chm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("big,small,nrhs", [(16384, 8192, 64), (8193, 8192, 64), (9000, 4096, 40), (8192, 8191, 33)])
def test_smaller_solve_allocates_nothing(big, small, nrhs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    chm.load(build_if_missing=True)
    L = torch.eye(big, dtype=torch.float32, device="cuda") * 2
    Ls = torch.eye(small, dtype=torch.float32, device="cuda") * 2
    B = torch.ones((nrhs, big), dtype=torch.float32, device="cuda")
    Bs = torch.ones((nrhs, small), dtype=torch.float32, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    assert chm.solve(L, B, stream=s) == chm.CHM_OK
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    assert chm.solve(Ls, Bs, stream=s) == chm.CHM_OK
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    assert chm.status_sync(s) == (chm.CHM_OK, -1)
    assert bool((B == 0.25).all()) and bool((Bs == 0.25).all())
