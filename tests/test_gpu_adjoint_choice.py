"""At l_max 2 the number of projections decides between the adjoint in channels
and in detector modes on volumes of more than a wave of voxel blocks: both sides
of that line against the FP64 handle (which always works in channels), with
rays that miss the detector.  FP32 positions and sums of a hundred terms:
1e-5 relative L2, the bound of every FP32 result."""
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_proj", [1, 31, 32])
@pytest.mark.parametrize("n_seg", [3, 8])
def test_l2_adjoint_on_both_sides(n_proj, n_seg):
    st = synth.small_setup(n=(70, 66, 83), nj=55, nk=61, ell_max=2, n_proj=n_proj, n_seg=n_seg, seed=n_proj)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    c = torch.randn(st.volume_shape, device="cuda", generator=gen)
    R = torch.randn(st.data_shape, device="cuda", generator=gen)
    h, h64 = tt.Handle(st, "f32"), tt.Handle(st, "f64")
    ref = h64.adjoint(R.double())
    assert float((h.adjoint(R).double() - ref).norm() / ref.norm()) <= 1e-5
    loss, g = h.gradient_residual(c, R)
    loss64, g64 = h64.gradient_residual(c.double(), R.double())
    assert abs(loss - loss64) <= 1e-5 * loss64
    assert float((g.double() - g64).norm() / g64.norm()) <= 1e-5
