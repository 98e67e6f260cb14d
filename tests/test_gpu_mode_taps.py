"""The forward in detector modes reads the taps that the other forwards read.
Seen with a NaN voxel in volumes whose rays run through voxel centres (no
rotation, no offset), where two of a ray's four taps per plane weigh nothing:
the rays that the voxel reaches are those of the FP64 handle."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ell", [6, 8])
@pytest.mark.parametrize("turned", [False, True])
@pytest.mark.parametrize("voxel", [(20, 15, 26), (21, 14, 27), (0, 0, 0), (40, 29, 52)])
def test_a_nan_voxel_reaches_the_same_rays(ell, turned, voxel):
    st = synth.small_setup(n=(41, 30, 53), nj=30, nk=41, ell_max=ell, n_proj=50, n_seg=8, seed=24, offsets=turned)
    if not turned:
        st = dataclasses.replace(st, inner_angle=np.zeros(50), outer_angle=np.zeros(50))
    h, ref = tt.Handle(st, "f32"), tt.Handle(st, "f64")
    c = torch.randn(st.volume_shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    c[voxel][0] = float("nan")
    bad, bad64 = torch.isnan(h.project(c)), torch.isnan(ref.project(c.double()))
    assert bad64.any() and torch.equal(bad, bad64)
