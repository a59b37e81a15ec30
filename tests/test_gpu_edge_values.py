"""Operators at the edges of their number range and of their launch limits.

Weights that are exactly zero beside values that are not finite, sums that leave the FP32 range on the
way to a result within it, infinities, rays that run along the edge of the frame, very many frames.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ops as O
from paper_2501_12497_gb300 import api, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def _out(fn, p, n, dtype, *args):
    out = torch.full((n,), float("nan"), device="cuda", dtype=dtype)
    fn(p, *args, out)
    return out


# A view at 0 degrees whose bin coordinates are whole numbers: the bin one footprint away from a pixel has
# the weight zero exactly (footprints within one bin, and within two).
@pytest.mark.parametrize("nb,db", [(60, 1.0), (61, 0.5)])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_fp64_transpose_takes_no_bin_of_weight_zero(nb, db, bad):
    n, ang = synth.shifted_angles(2, 3)
    assert ang[0] == 0.0
    p = api.mof_problem_create(40, 36, 2, nb, n, ang, 1.0, db, api.MOF_FP64)
    d = torch.ones(p.m, dtype=torch.float64, device="cuda")
    e = torch.zeros_like(d)
    d[15], e[15] = bad, 1.0
    out, foot = (_out(api.mof_apply_AT, p, p.n, torch.float64, v) for v in (d, e))
    assert (foot > 0).any()
    assert torch.equal(~torch.isfinite(out), foot > 0)
    if bad == float("inf"):
        assert not torch.isnan(out).any()


# A pixel's own terms may sum to more than FLT_MAX and be brought back by the scattered ones. The sums are
# taken in fixed point relative to the tile's largest term, so data scaled by a power of two give the
# same result scaled, bit for bit. Displacements within a few pixels (32-bit sums) and of up to 20 (64-bit).
@pytest.mark.parametrize("reach", [0.0, 2.0, 20.0])
def test_fp32_warp_transposes_near_the_largest_numbers(reach):
    p = api.mof_problem_create(70, 45, 4, 8, [1] * 4, np.zeros(4), 1.0, 1.0, api.MOF_FP32)
    g = torch.Generator(device="cuda").manual_seed(3)
    rand = lambda n, a: (torch.rand(n, device="cuda", generator=g) * 2 - 1) * a
    s, sr = rand(p.nv, reach), rand(p.nv, reach)
    down, up = 2.0 ** -8, 2.0 ** 8
    f32 = torch.float32

    r = rand(p.nv, 3.4e38)
    got, want = (_out(lambda q, v, o: api.mof_apply_flowT(q, v, s, sr, o), p, p.n, f32, v) for v in (r, r * down))
    assert torch.isfinite(got).float().mean() > 0.5
    assert torch.equal(got, want * up)

    x, uk = rand(p.n, 8e37), torch.zeros(p.n, device="cuda")
    got, want = (_out(lambda q, v, o: api.mof_apply_reg_normal(q, v, uk, s, sr, 1.0, o), p, p.n, f32, v) for v in (x, x * down))
    assert torch.isfinite(got).float().mean() > 0.5
    assert torch.equal(got, want * up)


# Infinities and overflow in the FP32 fan pair come out as infinities, as a plain sum has them. The views
# fill one stage of the transpose and several; the rays are marched in segments and whole.
@pytest.mark.parametrize("na,nb", [(9, 90), (40, 90), (800, 400)])
def test_fp32_fan_pair_keeps_infinities(na, nb):
    f32 = torch.float32
    p = api.mof_problem_create(64, 48, 2, nb, [na] * 2, 0.1234 + np.linspace(0, 3, 2 * na), 1.0, 1.6 * 90 / nb, api.MOF_FP32,
                               fan=(140.0, 70.0))
    g = torch.Generator(device="cuda").manual_seed(4)
    for fn, nin, nout, at in ((api.mof_apply_A, p.n, p.m, 64 * 20 + 30), (api.mof_apply_AT, p.m, p.n, 2 * nb + nb // 2)):
        x, e = torch.randn(nin, device="cuda", generator=g), torch.zeros(nin, device="cuda")
        x[at], e[at] = float("inf"), 1.0
        out, foot = (_out(fn, p, nout, f32, v) for v in (x, e))
        assert (foot > 0).any()
        assert torch.equal(torch.isinf(out), foot > 0) and not torch.isnan(out).any()
        out = _out(fn, p, nout, f32, torch.full((nin,), 3e38, device="cuda"))
        assert torch.isinf(out).any() and not torch.isnan(out).any()


# More frame pairs than one launch dimension holds: each pair's fields are those of the same frames in
# a short sequence. 4 columns: vectors of a row; 3: single pixels.
@pytest.mark.parametrize("nx", [4, 3])
@pytest.mark.parametrize("prec", [api.MOF_FP32, api.MOF_FP64])
def test_velocity_fields_of_very_many_frames(prec, nx):
    dt = torch.float64 if prec == api.MOF_FP64 else torch.float32
    ny, nt, few = 3, 65536 + 40, 9
    create = lambda t: api.mof_problem_create(nx, ny, t, 1, [1] * t, np.zeros(t), 1.0, 1.0, prec)
    p, q = create(nt), create(few)
    ns = nx * ny
    u = torch.randn(nt * ns, device="cuda", dtype=dt, generator=torch.Generator(device="cuda").manual_seed(5))
    fields = [torch.full(((nt - 1) * ns,), float("nan"), device="cuda", dtype=dt) for _ in range(3)]
    api.mof_of_fields(p, u, 1, *fields)
    assert all(torch.isfinite(f).all() for f in fields)
    for t0 in (0, 65530, 65535, nt - few):
        part = [torch.empty((few - 1) * ns, device="cuda", dtype=dt) for _ in range(3)]
        api.mof_of_fields(q, u[t0 * ns:(t0 + few) * ns].clone(), 1, *part)
        for f, want in zip(fields, part):
            assert torch.equal(f[t0 * ns:(t0 + few - 1) * ns], want)


# The last of 65 bins (by itself in its warp) looks along the frame's last column (row) from 2e-5 pixels
# inside, parallel to it and turned by up to 1e-6 rad, over a frame that is one in its outer columns (rows)
# only. A step's coordinate is exact to 2^-22 pixels and a ray takes 1024 of them; 1.5 times that is allowed.
def test_fp32_rays_along_the_edge_of_the_frame():
    n, nb, db, turns = 1024, 65, 512.49998 / 32, [0.0, 1e-6, -1e-6, 3e-7, -3e-7, 1e-7]
    ang = np.array(turns + [np.pi / 2 + a for a in turns])
    na = [len(turns)] * 2
    p = api.mof_problem_create(n, n, 2, nb, na, ang, 1.0, db, api.MOF_FP32)
    u = np.zeros((2, n, n))
    u[0, :, [0, -1]] = 1.0
    u[1, [0, -1], :] = 1.0
    want = O.project(O.Geometry(n, n, 2, nb, na, ang, 1.0, db), u).ravel()
    got = _out(api.mof_apply_A, p, p.m, torch.float32, torch.tensor(u.ravel(), device="cuda", dtype=torch.float32))
    assert (want.reshape(-1, nb)[:, -1] > 0.02).all()
    err = np.abs(got.cpu().numpy() - want).max()
    assert err <= 1.5 * n * 2.0 ** -22, err
