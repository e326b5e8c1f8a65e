"""The wave kernel where the rules send work to it: double factors above the
team kernel's range (here with a ragged order, an odd leading dimension and both
signs, in the bounds-checked build too and with a wait that runs out), plans of one
such factor, float factors above its range where path 1 is asked for, and one
vector into a large double factor in page-locked host memory.

Tolerances as in tests/common.py: float64 column-scaled 1e-11 against the
oracle's CholeskyModifyB, float the derived bound against its mixed emulation."""
from __future__ import annotations

import contextlib
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest
import torch

import oracle
from paper_1011_1173_gb300 import chm, inputs
from tests.common import TOL_F64, colscaled_err, tol_mixed

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    chm.load(build_if_missing=True)
    torch.cuda.set_device(0)
    yield
    chm.config_set("path", chm.PATH_AUTO)


def problem(n, k, pad, dtype=torch.float64):
    L = torch.full((n, n + pad), float("nan"), dtype=dtype, device="cuda")
    L[:, :n] = inputs.random_factor(n, 3, device="cuda", dtype=dtype)
    V = inputs.update_block(n, k, 3, device="cuda", dtype=dtype) * (0.5 / np.sqrt(n * k))
    return L, V, inputs.sigma_vector(k, 5)


def expected(L, V, sig, n):
    """The oracle's factor and the tolerance."""
    ref, k = L[:, :n].contiguous().cpu().numpy(), V.shape[0]
    if L.dtype == torch.float64:
        assert oracle.modify_b(ref, V.cpu().numpy(), sig.numpy())[0] == 0
        return ref, TOL_F64
    assert oracle.modify_mixed32(ref, V.cpu().numpy(), sig.numpy(), group=min(k, 64))[0] == 0
    return ref, tol_mixed(n, k)


@pytest.mark.parametrize("n,k,pad,dtype", [(6200, 17, 1, torch.float64), (8217, 3, 2, torch.float32)])
def test_ragged_padded_mixed_signs(n, k, pad, dtype):
    if dtype == torch.float64:
        assert chm.path_for(n, k, chm.CHM_F64) == chm.PATH_WAVE
    chm.config_set("path", chm.PATH_WAVE)
    L0, V, sig = problem(n, k, pad, dtype)
    ref, tol = expected(L0, V, sig, n)
    low = torch.ones((n, n), dtype=torch.bool, device="cuda").triu_(1)
    for checked in (False, True):
        L = L0.clone()
        with chm.checked_library() if checked else contextlib.nullcontext():
            chm.config_set("path", chm.PATH_WAVE)
            assert chm.modify(L, V, sig.tolist(), n=n) == chm.CHM_OK
            assert chm.status_sync() == (chm.CHM_OK, -1)
            if checked:
                chm.config_set("check_cut", 2)
                assert chm.modify(L0.clone(), V, sig.tolist(), n=n) == chm.CHM_OK
                st = chm.status_sync()[0]
                chm.config_set("check_cut", 0)
                chm.config_set("path", chm.PATH_AUTO)
                assert st == chm.CHM_ERR_BOUNDS
        assert torch.all(torch.isnan(L[:, n:]))
        assert torch.equal(L[:, :n][low], L0[:, :n][low])
        assert colscaled_err(L[:, :n].cpu().numpy(), ref) <= tol


def test_plan_of_one_factor_equals_the_call():
    n, k = 6200, 17
    L, V, _ = problem(n, k, 0)
    solo = L.clone()
    assert chm.modify(solo, V, 1) == chm.CHM_OK
    plan = chm.BatchPlan([n], [n], [k])
    assert plan.execute([L], [V]) == chm.CHM_OK
    assert plan.status() == (chm.CHM_OK, [(chm.CHM_OK, -1)])
    assert torch.equal(L, solo)
    before = L.clone()
    assert plan.autotune() == chm.CHM_OK and torch.equal(L, before)
    assert plan.execute([L], [V]) == chm.CHM_OK and chm.modify(solo, V, 1) == chm.CHM_OK
    assert plan.status()[0] == chm.CHM_OK and torch.equal(L, solo)
    plan.close()


def test_one_vector_into_a_host_factor():
    n = 8001
    L, V, sig = problem(n, 1, 1)
    ref, tol = expected(L, V, sig, n)
    host = torch.empty(L.shape, dtype=L.dtype, pin_memory=True).copy_(L)
    assert chm.modify(host, V, sig.tolist(), n=n) == chm.CHM_OK
    assert chm.status_sync() == (chm.CHM_OK, -1)
    assert colscaled_err(host[:, :n].numpy(), ref) <= tol


CHILD = textwrap.dedent("""
    import sys
    sys.path.insert(0, %r)
    import torch
    from paper_1011_1173_gb300 import chm, inputs
    chm.load(build_if_missing=True)
    n, k = 6200, 17
    L0 = inputs.random_factor(n, 3, device="cuda")
    V = inputs.update_block(n, k, 3, device="cuda") * 1e-3
    def run():
        L = L0.clone()
        assert chm.modify(L, V, 1) == chm.CHM_OK
        return chm.status_sync()[0], L
    assert run()[0] == chm.CHM_ERR_TIMEOUT
    a, b = run(), run()
    assert a[0] == b[0] == chm.CHM_OK and torch.equal(a[1], b[1])
    print("OK")
""" % ROOT)


def test_unreleased_panel_times_out():
    """As test_gpu_timeout, on the wave kernel."""
    env = dict(os.environ, CHM_TIMEOUT_NS=str(200_000_000), CHM_TEST_SKIP_PUBLISH="3")
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "OK" in r.stdout, r.stderr[-2000:]
