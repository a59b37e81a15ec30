"""The small projected solver called directly (mof::launch_small_solve), for calls that the
public entry points do not make at will."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_12497_gb300 import api

P, I, D = ctypes.c_void_p, ctypes.c_int, ctypes.c_double


class SmallArgs(ctypes.Structure):  # csrc/solver.cuh
    _fields_ = ([(n, P) for n in ("GA", "GL", "g", "bb", "K", "active")] + [(n, I) for n in ("ld", "B", "rule")] +
                [("target2", D), ("lam_fixed", D)] +
                [(n, P) for n in ("lam", "z", "flag", "err", "Mg", "Linv", "nL", "proj", "Y", "Yd", "Yh", "Yrho", "nY")])


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    return api.load()


def _launch(lib, args):
    fn = lib["_ZN3mof18launch_small_solveERKNS_9SmallArgsEP11CUstream_st"]
    fn.argtypes, fn.restype = [ctypes.POINTER(SmallArgs), P], I
    return fn(ctypes.byref(args), None)


# Bordered problems whose new eigenvalue all but coincides with an old one that hardly takes part: the
# FP32 search for a root can then stop on the wrong side of the pole by the FP32 rounding of the other
# terms (about 1e-8), and the FP64 step from there leaves the root's interval. Eigenvalues within 1e-11 (they
# lie in [0, 1]; each comes from sums of a few terms of up to a few tens, 1e-14, divided by a
# derivative of at least 1), and Y^T (G_A + rho G_L) Y = I, Y^T G_A Y diagonal within 1e-10.
@pytest.mark.gpu
def test_every_root_of_the_bordered_problem_is_found(lib):
    B, n = 4096, 4
    g = np.random.default_rng(7)
    a, b = g.uniform(-0.05, 0.05, B), g.uniform(-0.05, 0.05, B)
    d = np.stack([0.2 + a, 0.5 + b, 0.8 - a - b], 1)  # sum 3/2: G_A and I - G_A have equal traces, rho = 1
    c = np.stack([0.1 * g.uniform(0.5, 1.5, B), 10 ** g.uniform(-14, -10, B), 0.1 * g.uniform(0.5, 1.5, B)], 1)
    gam = d[:, 1] - c[:, 0] ** 2 / (d[:, 1] - d[:, 0]) - c[:, 2] ** 2 / (d[:, 1] - d[:, 2]) + 10 ** g.uniform(-8, -7.3, B)
    GA = np.zeros((B, n, n))
    GA[:, range(3), range(3)], GA[:, :3, 3], GA[:, 3, :3], GA[:, 3, 3] = d, c, c, gam
    GL = np.eye(n) - GA
    rhs = GA @ g.standard_normal((B, n, 1)) + 0.01 * g.standard_normal((B, n, 1))
    dev = lambda x, t=torch.float64: torch.tensor(x, device="cuda", dtype=t)
    zeros = lambda *s, t=torch.float64: torch.zeros(s, device="cuda", dtype=t)
    i32 = torch.int32
    T = dict(GA=dev(GA), GL=dev(GL), g=dev(rhs), bb=dev(np.full(B, 100.0)), K=dev(np.full(B, 3), i32), lam=zeros(B), z=zeros(B, n),
             flag=zeros(B, t=i32), err=zeros(1, t=i32), Y=zeros(B, n, n), Yd=zeros(B, n), Yh=zeros(B, n), Yrho=zeros(B),
             nY=zeros(B, t=i32))
    args = SmallArgs(ld=n, B=B, rule=api.MOF_RULE_GCV, **{k: v.data_ptr() for k, v in T.items()})
    torch.cuda.synchronize()
    for size in (3, 4):
        T["K"].fill_(size)
        torch.cuda.synchronize()
        assert _launch(lib, args) == api.MOF_OK
    torch.cuda.synchronize()
    assert int(T["err"]) == 0 and bool((T["nY"] == n).all())
    rho, got = T["Yrho"].cpu().numpy(), np.sort(T["Yd"].cpu().numpy(), 1)
    # of the pencil (G_A, G_A + rho G_L), rho = 1 but for a rounding
    M = GA + rho[:, None, None] * GL
    L = np.linalg.cholesky(M)
    C = np.linalg.solve(L, np.linalg.solve(L, GA).transpose(0, 2, 1))
    assert np.abs(got - np.linalg.eigvalsh(C)).max() <= 1e-11
    Y, Yd = T["Y"].cpu().numpy(), T["Yd"].cpu().numpy()
    Yt = Y.transpose(0, 2, 1)
    assert np.abs(Yt @ M @ Y - np.eye(n)).max() <= 1e-10
    assert np.abs(Yt @ GA @ Y - Yd[:, :, None] * np.eye(n)).max() <= 1e-10


# The state of a growing basis (Y) goes with the GCV rule only: the other rules leave parts of it unset.
@pytest.mark.parametrize("rule", [api.MOF_RULE_DP, api.MOF_RULE_FIXED])
def test_the_state_of_a_growing_basis_is_refused_with_other_rules(lib, rule):
    buf = (ctypes.c_double * 64)()
    at = ctypes.addressof(buf)
    args = SmallArgs(ld=4, B=0, rule=rule, Y=at)  # no problem: nothing could run
    assert _launch(lib, args) == api.MOF_EINVAL
