"""Segments of any width.  The basis matrix is formed by a 32-node rule, which is
not the exact mean of an order-8 harmonic over several turns; the detector modes
have to factor the matrix as it is formed, so projection and adjoint stay each
other's transpose.  Against the FP64 handle, which works in channels: 1e-5
relative L2, the FP32 bound of the parity tests."""
import dataclasses
import math

import numpy as np
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu
TOL = 1e-5


def rel(a, b):
    return float((a.double() - b).norm() / b.norm())


# the last size is one whose forward goes through modes
@pytest.mark.parametrize("ell,n_seg,n,n_proj", [(2, 4, (12, 11, 13), 19), (4, 6, (12, 11, 13), 19), (8, 10, (12, 11, 13), 21),
                                                (8, 10, (41, 40, 44), 48)])
@pytest.mark.parametrize("turns", [0.5, 1.0, 2.0, 3.0, 5.0])
def test_wide_segments(ell, n_seg, n, n_proj, turns):
    st = synth.small_setup(n=n, nj=n[1] + 2, nk=n[0] + 1, ell_max=ell, n_proj=n_proj, n_seg=n_seg, seed=3)
    s0 = np.linspace(0.1, 1.0, n_seg)
    st = dataclasses.replace(st, seg_start=s0, seg_end=s0 + 2.0 * math.pi * turns)
    h, ref = tt.Handle(st, "f32"), tt.Handle(st, "f64")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    c = torch.randn(st.volume_shape, device="cuda", generator=gen)
    R = torch.randn(st.data_shape, device="cuda", generator=gen)
    assert rel(h.project(c), ref.project(c.double())) <= TOL
    assert rel(h.adjoint(R), ref.adjoint(R.double())) <= TOL
    loss, g = h.gradient_residual(c, R)
    loss64, g64 = ref.gradient_residual(c.double(), R.double())
    assert abs(loss - loss64) <= TOL * loss64 and rel(g, g64) <= TOL
