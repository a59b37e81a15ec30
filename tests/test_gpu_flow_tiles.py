"""The tiled flow operators where their tiling and their choice of path can go wrong, against the
FP64 oracle: frames smaller than a tile and one pixel past it, displacements that vary by more
pixels than the short lists of the transposes hold, pixels that many sources reach, clipped
samples, rounded warps, and strips of the derivative fields with remainders.

Bars: an FP32 transpose sums its terms exactly, so it carries the roundings of three products per
term (2^-24 each) and one of the result: 1e-6 norm-wise; the derivative fields add up to 18 terms
of the frames' size: their error is held to 18 * 2^-24 of the largest frame value; the reverse
flow is bit-exact.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ops as O
from oracle import solver as OS
from paper_2501_12497_gb300 import api

pytestmark = pytest.mark.gpu

SHAPES = [(2, 2, 2), (63, 15, 2), (65, 17, 3), (64, 16, 2), (130, 33, 3), (36, 70, 2), (128, 67, 2)]
FIELDS = ["small", "spread", "sink", "out"]


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def _problem(shape, prec):
    nx, ny, nt = shape
    return api.mof_problem_create(nx, ny, nt, 1, [1] * nt, [0.0] * nt, precision=prec)


def _velocity(shape, kind, rng):
    nx, ny, nt = shape
    v = rng.uniform(-1.3, 1.3, (nt - 1, 2, ny, nx))
    if kind == "spread":  # displacements all over the frame
        v *= max(nx, ny)
    elif kind == "sink":  # every source goes to one pixel (up to its fraction)
        y, x = np.mgrid[0:ny, 0:nx]
        v[:, 0] = nx // 2 - x + 0.25 * rng.uniform(-1, 1, x.shape)
        v[:, 1] = ny // 2 - y + 0.25 * rng.uniform(-1, 1, x.shape)
    elif kind == "out":  # clipped at the frame's edges
        v[:, 0] += 5.0
        v[:, 1] -= 4.0
    return v


def _dev(a, prec):
    return torch.tensor(np.ascontiguousarray(a).ravel(), device="cuda", dtype=torch.float64 if prec == api.MOF_FP64 else torch.float32)


def _host(t):
    return t.cpu().double().numpy()


def _rel(a, b):
    return np.linalg.norm(a - np.ravel(b)) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("prec", [api.MOF_FP32, api.MOF_FP64])
@pytest.mark.parametrize("kind", FIELDS)
@pytest.mark.parametrize("shape", SHAPES)
def test_transposes_and_reverse_flow(shape, kind, prec):
    nx, ny, nt = shape
    rng = np.random.default_rng(nx * 7 + ny)
    p = _problem(shape, prec)
    s, sr = _dev(_velocity(shape, kind, rng), prec), _dev(_velocity(shape, "small", rng), prec)
    r = _dev(rng.standard_normal(2 * (nt - 1) * nx * ny), prec)
    x, uk = _dev(rng.standard_normal(nt * nx * ny), prec), _dev(rng.standard_normal(nt * nx * ny), prec)
    hs, hsr = (_host(v).reshape(nt - 1, 2, ny, nx) for v in (s, sr))
    hr = _host(r).reshape(2, nt - 1, ny, nx)
    bar = 1e-6 if prec == api.MOF_FP32 else 1e-13
    out = torch.full_like(x, float("nan"))
    api.mof_apply_flowT(p, r, s, sr, out)
    assert _rel(_host(out), O.flowT(hr, hs, hsr)) <= bar
    api.mof_apply_flowT(p, r, sr, s, out)
    assert _rel(_host(out), O.flowT(hr, hsr, hs)) <= bar
    # Theta^T W Theta: the weights 1 / sqrt(nu^2 + eps^2) of eps = 0.5 pass the rows' errors on at most 2-fold
    api.mof_apply_reg_normal(p, x, uk, s, sr, 0.5, out)
    th = OS.Theta((nt, ny, nx), hs, hsr)
    nu = th(_host(uk))
    assert _rel(_host(out), th.T(th(_host(x)) / np.sqrt(nu * nu + 0.25))) <= 4 * bar
    rev = torch.full_like(s, float("nan"))
    api.mof_reverse_flow(p, s, rev)
    want = O.reverse_flow(hs)
    want = want.astype(np.float32).astype(np.float64) if prec == api.MOF_FP32 else want
    assert np.array_equal(_host(rev), want.ravel())


def test_non_finite_term_stays_in_its_tiles():
    """A NaN source value makes the tiles that it reaches NaN; tiles out of its reach keep their values."""
    shape = (200, 50, 2)
    p = _problem(shape, api.MOF_FP32)
    rng = np.random.default_rng(3)
    s, sr = (_dev(_velocity(shape, "small", rng), api.MOF_FP32) for _ in range(2))
    r = _dev(rng.standard_normal(2 * 200 * 50), api.MOF_FP32)
    a, b = torch.empty(2 * 200 * 50, device="cuda"), torch.empty(2 * 200 * 50, device="cuda")
    api.mof_apply_flowT(p, r, s, sr, a)
    r[20 * 200 + 30] = float("nan")  # row r0 of the pair: own term of frame 0, scattered into frame 1
    api.mof_apply_flowT(p, r, s, sr, b)
    a, b = (v.cpu().numpy().reshape(2, 50, 200) for v in (a, b))
    assert np.isnan(b[:, 16:32, :64]).all()
    assert np.array_equal(a[:, :, 128:], b[:, :, 128:]) and np.array_equal(a[:, 48:], b[:, 48:])


@pytest.mark.parametrize("prec", [api.MOF_FP32, api.MOF_FP64])
@pytest.mark.parametrize("shape", [(2, 2, 2), (4, 3, 2), (33, 65, 3), (132, 70, 2), (257, 5, 2), (1024, 9, 3)])
def test_derivative_fields_in_strips(shape, prec):
    nx, ny, nt = shape
    p = _problem(shape, prec)
    u = _dev(np.random.default_rng(5).standard_normal((nt, ny, nx)), prec)
    f = [torch.full(((nt - 1) * ny * nx,), float("nan"), device="cuda", dtype=u.dtype) for _ in range(3)]
    api.mof_of_fields(p, u, 1, *f)
    want = O.of_fields(_host(u).reshape(nt, ny, nx), 1)
    tol = 18 * (2.0 ** -24 if prec == api.MOF_FP32 else 2.0 ** -53) * np.abs(_host(u)).max()
    for a, b in zip(f, want):
        assert np.max(np.abs(_host(a) - np.ravel(b))) <= tol
