"""Differentiable forms of the MMGKS-OF operators for torch.autograd.

Each forward and each backward pass is one or two calls into the C ABI (hand-written
sm_103a kernels); the nodes that allocate outputs and route gradients are native
(csrc/autograd.cpp):

  project(p, u)               b = H u                      (Sec. 2.1)
      backward: du = H^T db                                 (mof_apply_AT)
  flow_residual(p, u, s, sr)  r = Mhat(s, s') u            (Sec. 2.3, Sec. 3)
      backward: du  = Mhat(s, s')^T dr                      (mof_apply_flowT)
                ds, dsr = velocity VJP of Mhat(s, s') u      (mof_apply_flow_ds)

The velocity derivative is that of the clipped bilinear warp: the bilinear
slope on the forward pass's cell, zero along an axis where the sample point is
clipped (derivative from the right at integer sample positions). Tensors are
CUDA tensors of the problem's precision, flat or of any shape with the
problem's element counts; gradients come back flat.
"""
import importlib.util
import os

import torch

from . import api
from .build import AUTOGRAD_PATH

_native = None


def _nodes():
    global _native
    if _native is None:
        api.load()
        if not os.path.exists(AUTOGRAD_PATH):
            raise RuntimeError("_autograd.so is not built (%s); run __graft_entry__.build()" % AUTOGRAD_PATH)
        spec = importlib.util.spec_from_file_location("_autograd", AUTOGRAD_PATH)
        mod = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(mod)
        _native = mod
    return _native


def _dtype(p):
    return torch.float64 if p.precision == api.MOF_FP64 else torch.float32


def project(p, u):
    """H u for a problem p, differentiable in u."""
    if u.dtype != _dtype(p):
        raise TypeError("u must be %s for this problem" % _dtype(p))
    return _nodes().project(p, u)


def flow_residual(p, u, s, sr):
    """Mhat(s, s') u for a problem p, differentiable in u, s and sr."""
    for name, t in (("u", u), ("s", s), ("sr", sr)):
        if t.dtype != _dtype(p):
            raise TypeError("%s must be %s for this problem" % (name, _dtype(p)))
    return _nodes().flow_residual(p, u, s, sr)
