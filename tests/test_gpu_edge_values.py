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
