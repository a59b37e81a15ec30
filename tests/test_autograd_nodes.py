"""The native autograd nodes: what they refuse, and the lifetime of what they hold."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_12497_gb300 import api
from paper_2501_12497_gb300 import autograd as AG


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


class _Sizes:  # the attributes of a problem that the nodes read
    handle, n, m, nv, precision = ctypes.c_void_p(0), 4, 3, 2, api.MOF_FP32


def test_refused_before_the_gpu_is_touched():
    p, z = _Sizes(), torch.zeros
    with pytest.raises(ValueError, match="u must be a CUDA tensor"):
        AG.project(p, z(4))
    with pytest.raises(ValueError, match="u must be a CUDA tensor"):
        AG.flow_residual(p, z(4, requires_grad=True), z(2), z(2))
    with pytest.raises(TypeError, match="u must be torch.float32"):
        AG.project(p, z(4, dtype=torch.float64))
    with pytest.raises(TypeError, match="sr must be torch.float32"):
        AG.flow_residual(p, z(4), z(2), z(2, dtype=torch.float64))


def _problem():
    return api.mof_problem_create(20, 18, 3, 30, [4] * 3, np.linspace(0, 3, 12), 1.0, 1.0, api.MOF_FP32)


@pytest.mark.gpu
def test_problem_lifetime_and_status():
    p = _problem()
    u = torch.rand(p.n, device="cuda", requires_grad=True)
    want = torch.empty(p.n, device="cuda")
    db = torch.rand(p.m, device="cuda")
    api.mof_apply_AT(p, db, want)
    b = AG.project(p, u)
    with pytest.raises(ValueError, match="u has 5 elements, expected %d" % p.n):
        AG.project(p, u[:5])
    del p  # held by the graph
    b.backward(db, retain_graph=True)
    assert torch.equal(u.grad, want)
    q = _problem()
    b = AG.project(q, u)
    q.close()
    with pytest.raises(api.MofError):
        b.backward(db)
    with pytest.raises(api.MofError):
        AG.project(q, u)


@pytest.mark.gpu
def test_layouts_parts_and_streams():
    p = _problem()
    g = torch.Generator(device="cuda").manual_seed(1)
    r = lambda n: torch.randn(n, device="cuda", generator=g)
    u, s, sr = r(p.n), r(p.nv), r(p.nv)
    dr = r(p.nv)
    want, gs, gsr, gu = (torch.empty(n, device="cuda") for n in (p.nv, p.nv, p.nv, p.n))
    api.mof_apply_flow(p, u, s, sr, want)
    api.mof_apply_flowT(p, dr, s, sr, gu)
    api.mof_apply_flow_ds(p, u, s, sr, dr, gs, gsr)
    # strided input and cotangent, a gradient of one input only, another stream
    u2 = torch.stack([u, u], 1)[:, 0]
    s1 = s.clone().requires_grad_()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        out = AG.flow_residual(p, u2, s1, sr)
        (got,) = torch.autograd.grad(out, s1, torch.stack([dr, dr], 1)[:, 0])
    torch.cuda.current_stream().wait_stream(stream)
    assert torch.equal(out, want) and torch.equal(got, gs)
    u3, sr3 = u.clone().requires_grad_(), sr.clone().requires_grad_()
    out = AG.flow_residual(p, u3, s, sr3)
    a, c = torch.autograd.grad(out, (u3, sr3), dr)
    assert torch.allclose(a, gu, rtol=1e-5, atol=1e-6) and torch.equal(c, gsr)
    with torch.no_grad():
        assert not AG.project(p, u3).requires_grad
