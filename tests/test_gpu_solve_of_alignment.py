"""Solve-OF into a velocity array that no 16-byte vector store may be aimed at.

The plain form and a timed call write s where the caller has it (the graph form solves into the
workspace and copies): one element off a 16-byte boundary the same values have to arrive, and nothing
beside them.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_12497_gb300 import api, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


# 64 x 64: the one-pass projection; 45 x 47 (no multiple of 16 bytes): the general sequence
@pytest.mark.parametrize("nx,ny", [(64, 64), (45, 47)])
@pytest.mark.parametrize("timed", [False, True])
@pytest.mark.parametrize("prec", [api.MOF_FP32, api.MOF_FP64])
def test_velocities_one_element_off_a_vector_boundary(prec, timed, nx, ny):
    dt = torch.float64 if prec == api.MOF_FP64 else torch.float32
    y, x = np.mgrid[0:ny, 0:nx] / 64.0
    u = np.stack([np.sin(7 * x + 0.05 * t) * np.cos(5 * y - 0.04 * t) for t in range(4)])
    u = u + 0.01 * np.random.default_rng(1).standard_normal(u.shape)
    p = api.mof_problem_create(nx, ny, 4, 8, [1] * 4, np.zeros(4), 1.0, 1.0, prec)
    ud = torch.tensor(u, device="cuda", dtype=dt).reshape(-1)
    prm = api.mof_default_params(of_ell=4, of_iters=5, plain=0 if timed else 1)
    if timed:
        api.mof_set_timing(p, 1)
    want = torch.empty(p.nv, dtype=dt, device="cuda")
    assert want.data_ptr() % 16 == 0
    api.mof_solve_of(p, prm, ud, want)
    buf = torch.full((p.nv + 2,), 7.0, dtype=dt, device="cuda")
    s = buf[1:1 + p.nv]
    assert s.data_ptr() % 16 != 0
    api.mof_solve_of(p, prm, ud, s)
    assert torch.equal(s, want) and torch.isfinite(s).all() and float(s.abs().max()) > 0
    assert float(buf[0]) == 7.0 and float(buf[-1]) == 7.0
