"""Waits that run out for some tiles and not for others.

With a bound of a few polls some warps of Solve-OF's projection pass get their tile in time and
others, or the same ones at a later tile, do not: the call returns with its result or with MOF_ETIMEOUT, and
the next call with the default bound gives the result it gave before, bit for bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_12497_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


# 362 x 362 pixels, 10 pairs: two tiles per warp in FP32, four in FP64
@pytest.mark.parametrize("polls", [1, 4])
@pytest.mark.parametrize("prec", [api.MOF_FP32, api.MOF_FP64])
def test_waits_that_run_out_here_and_there(prec, polls):
    n, nt = 362, 11
    dt = torch.float64 if prec == api.MOF_FP64 else torch.float32
    y, x = np.mgrid[0:n, 0:n] / n
    u = torch.tensor(np.stack([np.sin(7 * x + 0.05 * t) * np.cos(5 * y - 0.04 * t) for t in range(nt)]), device="cuda", dtype=dt).reshape(-1)
    p = api.mof_problem_create(n, n, nt, 8, [1] * nt, np.zeros(nt), 1.0, 1.0, prec)
    prm = api.mof_default_params(of_ell=3, of_iters=4)
    want, got = (torch.empty(p.nv, dtype=dt, device="cuda") for _ in range(2))
    api.mof_solve_of(p, prm, u, want)
    try:
        api.mof_debug_set_wait_limit(polls)
        try:
            api.mof_solve_of(p, prm, u, got)
            assert torch.equal(got, want)
        except api.MofError as e:
            assert e.status == api.MOF_ETIMEOUT
    finally:
        api.mof_debug_set_wait_limit(-1)
    api.mof_solve_of(p, prm, u, got)
    assert torch.equal(got, want)
