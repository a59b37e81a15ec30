"""The small problem of Solve-OF, updated from one iteration to the next by a bordered
eigenproblem, against the FP64 oracle at the sizes where its work is split differently.

The oracle searches lambda by golden section, which fixes log10(lambda) to ~1e-8, and solves by
QR and SVD: FP64 results agree to 1e-7 per solve, and 1e-6 is allowed over up to 63 of them.
FP32 operators carry 6e-8 per application into up to 63 iterations: the bar of 1e-3 that the
shorter solves have.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import solver as OS
from paper_2501_12497_gb300 import api, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


# basis sizes: from the first column; across 32 roots (two to four threads' parts per root);
# up to the largest, 64; a single iteration (no update at all)
@pytest.mark.parametrize("ell,iters", [(1, 6), (28, 9), (2, 62), (63, 1), (62, 2)])
@pytest.mark.parametrize("prec", [api.MOF_FP64, api.MOF_FP32])
def test_bordered_solves(prec, ell, iters):
    w = synth.moving_disks(40, 4, 8, 40, radii=(5.0, 8.0), seed=4)
    p = api.mof_problem_create(w.nx, w.ny, w.nt, w.nb, w.na, w.angles, w.h, w.db, prec)
    f64 = prec == api.MOF_FP64
    u = w.u_true.astype(np.float64 if f64 else np.float32).copy()
    u[2] = u[1]  # a pair without motion: nothing to solve beside pairs that do
    s = torch.empty(p.nv, dtype=torch.float64 if f64 else torch.float32, device="cuda")
    api.mof_solve_of(p, api.mof_default_params(of_ell=ell, of_iters=iters), torch.tensor(u, device="cuda").reshape(-1), s)
    want = OS.solve_of(u.astype(np.float64), OS.Params(of_ell=ell, of_iters=iters))
    got = s.cpu().double().numpy().reshape(want.shape)
    err = np.linalg.norm(got - want) / np.linalg.norm(want)
    assert err <= (1e-6 if f64 else 1e-3), err


# frames whose last tile of the projection pass is ragged, and enough of them that a warp takes
# several tiles (2 in FP32, 4 in FP64)
@pytest.mark.parametrize("prec", [api.MOF_FP64, api.MOF_FP32])
def test_projection_pass_tiles(prec):
    n, nt = 362, 11
    g = np.random.default_rng(5)
    f64 = prec == api.MOF_FP64
    y, x = np.mgrid[0:n, 0:n] / n
    u = np.stack([np.sin(7 * x + 0.05 * t) * np.cos(5 * y - 0.04 * t) for t in range(nt)]) + 0.01 * g.standard_normal((nt, n, n))
    u = u.astype(np.float64 if f64 else np.float32)
    p = api.mof_problem_create(n, n, nt, 8, [1] * nt, np.zeros(nt), 1.0, 1.0, prec)
    s = torch.empty(p.nv, dtype=torch.float64 if f64 else torch.float32, device="cuda")
    api.mof_solve_of(p, api.mof_default_params(of_ell=3, of_iters=6), torch.tensor(u, device="cuda").reshape(-1), s)
    want = OS.solve_of(u.astype(np.float64), OS.Params(of_ell=3, of_iters=6))
    got = s.cpu().double().numpy().reshape(want.shape)
    err = np.linalg.norm(got - want) / np.linalg.norm(want)
    assert err <= (1e-6 if f64 else 1e-3), err


# widths whose rows are taken by the marching residual kernel in strips of 4 rows (364 x 61: a last
# strip of one row, the last warp with one lane of its own) and of 16 (364 x 1000), frames that are no
# multiple of 4 values (45 x 47: scalar half-steps, no one-pass projection) and of many chunks
@pytest.mark.parametrize("nx,ny,nt,ell,iters", [(364, 61, 22, 3, 4), (364, 1000, 14, 2, 2), (45, 47, 5, 12, 3), (128, 65, 4, 9, 2)])
@pytest.mark.parametrize("prec", [api.MOF_FP64, api.MOF_FP32])
def test_residual_and_golub_kahan_sizes(prec, nx, ny, nt, ell, iters):
    g = np.random.default_rng(6)
    f64 = prec == api.MOF_FP64
    y, x = np.mgrid[0:ny, 0:nx] / max(nx, ny)
    u = np.stack([np.sin(9 * x + 0.05 * t) * np.cos(6 * y - 0.04 * t) for t in range(nt)]) + 0.01 * g.standard_normal((nt, ny, nx))
    u = u.astype(np.float64 if f64 else np.float32)
    p = api.mof_problem_create(nx, ny, nt, 8, [1] * nt, np.zeros(nt), 1.0, 1.0, prec)
    s = torch.empty(p.nv, dtype=torch.float64 if f64 else torch.float32, device="cuda")
    api.mof_solve_of(p, api.mof_default_params(of_ell=ell, of_iters=iters), torch.tensor(u, device="cuda").reshape(-1), s)
    want = OS.solve_of(u.astype(np.float64), OS.Params(of_ell=ell, of_iters=iters))
    got = s.cpu().double().numpy().reshape(want.shape)
    err = np.linalg.norm(got - want) / np.linalg.norm(want)
    assert err <= (1e-6 if f64 else 1e-3), err
