"""The FP32 projector pair at the sizes where its tiling can go wrong, against the FP64 oracle.

Sizes: frames smaller than a tile or a warp's rays, one pixel past a tile, segments of the steps
(few rays), more views than one stage holds, views at 0, 45 and 90 degrees, detectors up to twice
as fine as the pixels (staged footprints of one and of two bins each side), finer (the general
transpose) and much coarser than them.

Bar: a tap's weight is exact to 2^-22 (its coordinate) plus two roundings of 2^-24, against a
weight whose root mean square over a pixel is 1/sqrt(3) or more, and sums are compensated, so the
relative 2-norm error on random data stays below 2^-22 sqrt(3) + 3 * 2^-24 < 6e-7; 1e-6 is asserted.
A coarse detector scales a coordinate's error by 1/r (r the footprint in bins).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ops as O
from paper_2501_12497_gb300 import api, synth

pytestmark = pytest.mark.gpu

# nx, ny, nt, na, nb, bin size
CASES = [(2, 2, 2, 1, 1, 1.0), (3, 5, 2, 4, 9, 1.0), (31, 33, 2, 5, 32, 1.0), (33, 65, 3, 33, 97, 1.0), (64, 32, 2, 65, 33, 1.0),
         (130, 17, 2, 4, 190, 1.0), (96, 96, 2, 8, 271, 0.5), (65, 40, 2, 9, 160, 0.51), (40, 33, 2, 9, 160, 0.3),
         (50, 47, 2, 7, 31, 2.5), (257, 255, 2, 6, 363, 1.0)]


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def _pair(case, fan=None):
    nx, ny, nt, na, nb, db = case
    n, ang = synth.shifted_angles(nt, na)
    p = api.mof_problem_create(nx, ny, nt, nb, n, ang, 1.0, db, api.MOF_FP32, fan=fan)
    return p, O.Geometry(nx, ny, nt, nb, n, ang, 1.0, db, fan=fan)


def _rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


def _apply(p, fn, x, n):
    out = torch.full((n,), float("nan"), device="cuda")
    fn(p, torch.tensor(x, device="cuda"), out)
    return out.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("case", CASES)
def test_pair_at_tile_edges(case):
    p, g = _pair(case)
    rng = np.random.default_rng(1)
    u, d = rng.standard_normal(p.n).astype(np.float32), rng.standard_normal(p.m).astype(np.float32)
    bar = 1e-6 * max(1.0, case[5])
    assert _rel(_apply(p, api.mof_apply_A, u, p.m), O.project(g, u.astype(np.float64)).ravel()) <= bar
    assert _rel(_apply(p, api.mof_apply_AT, d, p.n), O.backproject(g, d.astype(np.float64)).ravel()) <= bar


@pytest.mark.parametrize("case", [(33, 31, 2, 9, 64, 1.1), (130, 40, 2, 4, 200, 1.3)])
def test_fan_march_at_warp_edges(case):
    p, g = _pair(case, fan=(260.0, 60.0))
    u = np.random.default_rng(2).standard_normal(p.n).astype(np.float32)
    assert _rel(_apply(p, api.mof_apply_A, u, p.m), O.project(g, u.astype(np.float64)).ravel()) <= 1e-6


def test_rays_far_beyond_the_frame_see_nothing():
    """Bins a million pixels apart: only the middle bin's rays cross the frame."""
    p, g = _pair((40, 40, 2, 3, 9, 1e6))
    u = np.random.default_rng(3).standard_normal(p.n).astype(np.float32)
    b = _apply(p, api.mof_apply_A, u, p.m).reshape(-1, 9)
    assert np.all(b[:, [0, 1, 2, 3, 5, 6, 7, 8]] == 0)
    assert _rel(b.ravel(), O.project(g, u.astype(np.float64)).ravel()) <= 1e-6


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("db", [1.0, 0.6])
def test_non_finite_bin_reaches_its_own_footprint_only(db, bad):
    p, g = _pair((45, 45, 2, 5, 120, db))
    d = np.random.default_rng(4).standard_normal(p.m).astype(np.float32)
    k = 2 * 120 + 61  # a bin in the middle of the third view
    e = np.zeros(p.m)
    e[k] = 1.0
    w = O.backproject(g, e).ravel()
    want = _apply(p, api.mof_apply_AT, d, p.n)
    d[k] = bad
    out = _apply(p, api.mof_apply_AT, d, p.n)
    assert not np.isfinite(out[w > 1e-4]).any()
    assert np.array_equal(out[w == 0], want[w == 0])


# nx, ny, nt, na, nb, bin size, source and detector distance: the 1.5x magnification of the
# workloads on tiles with remainders (views beyond one stage, fans that straddle 45 degrees), the
# same turned to 45 degrees exactly, and a source too near for the tiled form
FANS = [(33, 65, 2, 17, 100, 1.6, 140.0, 70.0), (64, 64, 2, 4, 97, 1.5, 128.0, 64.0), (200, 31, 2, 5, 260, 1.6, 400.0, 200.0),
        (31, 31, 2, 33, 64, 1.2, 30.0, 3.0)]


@pytest.mark.parametrize("case", FANS)
def test_fan_transpose_at_tile_edges(case):
    nx, ny, nt, na, nb, db, rs, rd = case
    p, g = _pair((nx, ny, nt, na, nb, db), fan=(rs, rd))
    d = np.random.default_rng(5).standard_normal(p.m).astype(np.float32)
    assert _rel(_apply(p, api.mof_apply_AT, d, p.n), O.backproject(g, d.astype(np.float64)).ravel()) <= 1e-6


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_fan_non_finite_bin_reaches_its_own_rays_pixels_only(bad):
    p, g = _pair((64, 48, 2, 5, 100, 1.6), fan=(140.0, 70.0))
    d = np.random.default_rng(6).standard_normal(p.m).astype(np.float32)
    k = 3 * 100 + 52
    e = np.zeros(p.m)
    e[k] = 1.0
    w = O.backproject(g, e).ravel()
    want = _apply(p, api.mof_apply_AT, d, p.n)
    d[k] = bad
    out = _apply(p, api.mof_apply_AT, d, p.n)
    assert not np.isfinite(out[w > 1e-4]).any()
    assert np.array_equal(out[w == 0], want[w == 0])
