"""The staged forward takes rings up to its limit of 200 KB whatever the epilogue
needs beside them: detector axes at 45 degrees to the volume's and pixels of 1.87
voxels make boxes of 32 x 32 voxels, three of which and 64 segments' basis rows take
196 KB.  Projections and gradients are the tap-pair march's, bit for bit (the loss,
summed over other tiles, to 1e-6)."""
import dataclasses
import math

import numpy as np
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_proj", [2, 20])
def test_largest_ring(n_proj):
    s = math.sqrt(0.5)
    frame = dict(tt.STANDARD_FRAME, j=(s, s, 0.0), k=(s, -s, 0.0))
    st = synth.small_setup(n=(40, 38, 36), nj=18, nk=19, ell_max=4, n_proj=n_proj, n_seg=64, seed=1, b=1.87)
    st = dataclasses.replace(st, inner_angle=np.zeros(n_proj), outer_angle=np.zeros(n_proj))
    h, l1 = tt.Handle(st, "f32", frame=frame), tt.Handle(st, "f32", frame=frame)
    h.set_forward_kernel("staged")
    l1.set_forward_kernel("l1")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    c = torch.randn(st.volume_shape, device="cuda", generator=gen)
    I = torch.randn(st.data_shape, device="cuda", generator=gen)
    assert torch.equal(h.project(c), l1.project(c))
    loss, g = h.gradient_residual(c, I)
    loss1, g1 = l1.gradient_residual(c, I)
    assert torch.equal(g, g1) and abs(loss - loss1) <= 1e-6 * loss1
