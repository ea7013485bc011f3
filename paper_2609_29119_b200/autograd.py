"""Differentiable wrappers: transforms whose forward and backward are the library's own calls.

Under the real inner product <u, v> = Re(u^H v) (Sec. 3.2) the backward of the analysis T is the real adjoint
T^dagger (cqt_analyse_adjoint) applied to the coefficient cotangent, and the backward of the synthesis S is
S^dagger (cqt_synthesise_adjoint) applied to the signal cotangent.  That is PyTorch's convention for complex
tensors (the gradient of a real loss with respect to c is dL/dRe c + i dL/dIm c).  No transform activation is
saved: both backward passes need the cotangent only.  The autograd nodes are native (csrc/torch_ext.cpp).
"""
from .binding import ANALYSE, SYNTHESISE, native


def analyse(plan, x, valid_len=None):
    """c = T x with gradient support; x [batch, >= valid_len] float32 on the plan's device."""
    return native().differentiable(plan, ANALYSE, x, valid_len)


def synthesise(plan, c, valid_len=None):
    """x = S c with gradient support; c [batch, coeff_count] complex64 on the plan's device."""
    return native().differentiable(plan, SYNTHESISE, c, valid_len)
