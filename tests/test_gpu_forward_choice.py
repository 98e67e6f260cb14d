"""Which forward an automatic handle runs at l_max 6 and 8: the one in modes maps
the whole volume for every projection, so it is taken where enough rays cross it.
Seen by the launches of a projection (the direct march: one pack; modes: the maps
too), on both sides of the line: detectors as large as the volume, narrow ones,
ones that lie beside it, little work, 2-byte storage.  Both forwards agree with
the FP64 handle (1e-5 relative L2; 2-byte: as in the precision tests)."""
import dataclasses

import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu
TOL = {"f32": 1e-5, "bf16": 5e-3, "f16": 1e-3}

CASES = [  # volume, pixels, l_max, projections, precision, shift of the detector, modes?
    ((48, 40, 48), (40, 48), 6, 60, "f32", 0.0, True),
    ((48, 40, 48), (40, 48), 8, 60, "f32", 0.0, True),
    ((48, 40, 48), (8, 48), 6, 60, "f32", 0.0, False),
    ((48, 40, 48), (40, 9), 8, 60, "f32", 0.0, False),
    ((48, 40, 48), (40, 48), 8, 60, "f32", 30.0, False),
    ((48, 40, 48), (40, 48), 8, 60, "f32", 300.0, False),
    ((30, 24, 60), (90, 91), 8, 80, "f32", 0.0, True),
    ((24, 20, 24), (20, 24), 8, 60, "f32", 0.0, False),
    ((48, 40, 48), (40, 48), 4, 60, "f32", 0.0, False),
    ((64, 60, 64), (60, 64), 6, 120, "bf16", 0.0, False),
    ((64, 60, 64), (60, 64), 8, 120, "bf16", 0.0, True),
    ((64, 60, 64), (60, 64), 8, 120, "f16", 0.0, True),
    ((48, 40, 48), (40, 48), 8, 60, "f16", 0.0, False),
]


@pytest.mark.parametrize("n,pixels,ell,n_proj,prec,shift,modes", CASES)
def test_forward_by_the_rays_that_cross(n, pixels, ell, n_proj, prec, shift, modes):
    st = synth.small_setup(n=n, nj=pixels[0], nk=pixels[1], ell_max=ell, n_proj=n_proj, n_seg=8, seed=7)
    st = dataclasses.replace(st, j_offset=st.j_offset + shift)
    h, ref = tt.Handle(st, prec), tt.Handle(st, "f64")
    c = torch.randn(st.volume_shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
    h.profile(True)
    h.profile_reset()
    got = h.project(c)
    assert (h.profile_read()["pack"][1] > 1) == modes
    h.profile(False)
    want = ref.project(c.double())
    assert float((got.double() - want).norm()) <= TOL[prec] * float(want.norm())
