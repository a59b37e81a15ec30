"""The FP64 parallel-beam pair in fixed-point coordinates at its edges, against the FP64 oracle.

Frames smaller than a tile or a warp's rays, quarters of the steps that are empty, more views than
one stage holds, views at 0, 45 and 90 degrees, footprints within one and two bins each side, wider
ones and frames beyond the fixed-point range (the general kernels), rays that miss the frame.

Bar: both sides round a coordinate of at most 512 a few times, 4 x 2^-44 = 2.3e-13 bins or pixels at
most, against weights whose root mean square is 1/sqrt(3) or more: 1e-12 is asserted, scaled by the
detector's coarseness, and by 8 for the frame of 4001 pixels.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ops as O
from paper_2501_12497_gb300 import api, synth

pytestmark = pytest.mark.gpu

# nx, ny, nt, na, nb, bin size
CASES = [(2, 2, 2, 1, 1, 1.0), (3, 5, 2, 4, 9, 1.0), (31, 33, 2, 5, 32, 1.0), (33, 65, 3, 33, 97, 1.0), (64, 64, 2, 65, 64, 1.0),
         (130, 17, 2, 4, 190, 1.0), (96, 96, 2, 8, 271, 0.5), (40, 33, 2, 9, 160, 0.3), (50, 47, 2, 7, 31, 2.5),
         (257, 255, 2, 6, 363, 1.0), (40, 44, 2, 6, 400, 1.0), (4001, 3, 2, 3, 70, 60.0)]


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("case", CASES)
def test_fp64_pair_at_edges(case):
    nx, ny, nt, na, nb, db = case
    n, ang = synth.shifted_angles(nt, na)
    p, g = api.mof_problem_create(nx, ny, nt, nb, n, ang, 1.0, db, api.MOF_FP64), O.Geometry(nx, ny, nt, nb, n, ang, 1.0, db)
    rng = np.random.default_rng(1)
    u, d = rng.standard_normal(p.n), rng.standard_normal(p.m)
    bar = 1e-12 * max(1.0, db) * (8 if nx > 4000 else 1)
    for fn, x, size, want in ((api.mof_apply_A, u, p.m, O.project(g, u)), (api.mof_apply_AT, d, p.n, O.backproject(g, d))):
        out = torch.full((size,), float("nan"), device="cuda", dtype=torch.float64)
        fn(p, torch.tensor(x, device="cuda"), out)
        want = np.ravel(want)
        err = np.linalg.norm(out.cpu().numpy() - want) / max(np.linalg.norm(want), 1e-300)
        assert err <= bar, err


def test_fp64_values_that_are_not_finite_stay_in_their_footprint():
    n, ang = synth.shifted_angles(2, 3)
    p = api.mof_problem_create(40, 36, 2, 60, n, ang, 1.0, 1.0, api.MOF_FP64)
    d = torch.ones(p.m, dtype=torch.float64, device="cuda")
    e = torch.zeros_like(d)
    d[75], e[75] = float("inf"), 1.0
    out, foot = (torch.empty(p.n, dtype=torch.float64, device="cuda") for _ in range(2))
    api.mof_apply_AT(p, d, out)
    api.mof_apply_AT(p, e, foot)
    assert torch.equal(torch.isinf(out), foot > 0) and not torch.isnan(out).any()
