"""FP32 at l_max 6 (32 channels): grids that two CTAs per SM hold at once, that only
three do, and larger ones run with different numbers asked for.  A ray's bits do not
depend on it, and each agrees with the FP64 handle (1e-5 relative L2)."""
import dataclasses

import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_proj", [19, 20, 28, 29])   # of 16 tiles: 304 and 456 lie between
@pytest.mark.parametrize("n_seg", [4, 7])
def test_grids_by_their_waves(n_proj, n_seg):
    many = synth.small_setup(n=(30, 28, 31), nj=30, nk=32, ell_max=6, n_proj=n_proj, n_seg=n_seg, seed=3)
    few = dataclasses.replace(many, inner_angle=many.inner_angle[:5], outer_angle=many.outer_angle[:5],
                              j_offset=many.j_offset[:5], k_offset=many.k_offset[:5])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    c = torch.randn(many.volume_shape, device="cuda", generator=gen)
    I = torch.randn(many.data_shape, device="cuda", generator=gen)
    h, ref = tt.Handle(many, "f32"), tt.Handle(many, "f64")
    assert torch.equal(h.project(c)[:5], tt.Handle(few, "f32").project(c))
    loss, g = h.gradient_residual(c, I)
    loss64, g64 = ref.gradient_residual(c.double(), I.double())
    assert abs(loss - loss64) <= 1e-5 * loss64
    assert float((g.double() - g64).norm() / g64.norm()) <= 1e-5
