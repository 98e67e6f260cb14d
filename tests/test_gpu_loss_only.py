"""The loss without a gradient takes other kernels than an evaluation: it is the
evaluation's loss bit for bit where both march the volume (the sums of W r^2 do not
depend on what the residual is contracted to), and to FP32 rounding elsewhere."""
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "bf16", "f16", "f64"])
@pytest.mark.parametrize("ell,n,n_proj", [(2, (20, 18, 21), 30), (4, (20, 18, 21), 30), (8, (20, 18, 21), 30),
                                          (8, (56, 50, 56), 60), (10, (20, 18, 21), 9)])
def test_loss_alone(prec, ell, n, n_proj):
    st = synth.small_setup(n=n, nj=n[1] + 3, nk=n[0] + 1, ell_max=ell, n_proj=n_proj, n_seg=8, seed=ell)
    h = tt.Handle(st, prec)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    c = torch.randn(st.volume_shape, device="cuda", generator=gen).to(h.dtype)
    I = torch.randn(st.data_shape, device="cuda", generator=gen).to(h.dtype)
    W = torch.rand(st.data_shape, device="cuda", generator=gen).to(h.dtype)
    for w in (None, W):
        for vol in (c, None):
            loss, g = h.gradient_residual(vol, I, w)
            alone, none = h.gradient_residual(vol, I, w, want_grad=False)
            assert none is None and alone == loss
            again, g2 = h.gradient_residual(vol, I, w)
            assert again == loss and torch.equal(g, g2)
