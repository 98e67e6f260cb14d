"""The host-buffer entry point where the forward goes through modes (fewer, larger
chunks): the bits of the device entry point, pinned and pageable, with and without
weights."""
import numpy as np
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ell,n_proj", [(6, 47), (8, 50), (6, 130), (8, 245)])
@pytest.mark.parametrize("pinned", [False, True])
def test_host_equals_device(ell, n_proj, pinned):
    st = synth.small_setup(n=(44, 41, 45), nj=42, nk=43, ell_max=ell, n_proj=n_proj, n_seg=8, seed=n_proj)
    h = tt.Handle(st, "f32")
    gen = torch.Generator()
    gen.manual_seed(1)

    def host(shape):
        a = torch.rand(shape, generator=gen) - 0.3
        return a.pin_memory() if pinned else a

    c, I, W = host(st.volume_shape), host(st.data_shape), host(st.data_shape)
    for w in (None, W):
        out = host(st.volume_shape).numpy()
        loss, g = h.gradient_residual_host(c.numpy(), I.numpy(), None if w is None else w.numpy(), out)
        loss_d, g_d = h.gradient_residual(c.cuda(), I.cuda(), None if w is None else w.cuda())
        assert loss == loss_d and np.array_equal(g, g_d.cpu().numpy())
