"""The host-buffer entry point's chunks, one per 20 projections and eight at most: the
bits of the device entry point at the edges between numbers of chunks."""
import numpy as np
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,ell", [("f32", 2), ("f32", 4), ("f16", 4), ("bf16", 0)])
@pytest.mark.parametrize("n_proj", [1, 2, 19, 20, 39, 40, 41, 59, 61, 159, 160, 163])
def test_host_equals_device(prec, ell, n_proj):
    st = synth.small_setup(n=(18, 21, 17), nj=20, nk=23, ell_max=ell, n_proj=n_proj, n_seg=5, seed=n_proj)
    h = tt.Handle(st, prec)
    gen = torch.Generator()
    gen.manual_seed(1)
    c, I, W = (torch.rand(s, generator=gen) - 0.3 for s in (st.volume_shape, st.data_shape, st.data_shape))
    for pinned in (False, True):
        a, b, w = (t.pin_memory() if pinned else t for t in (c, I, W))
        out = torch.empty(st.volume_shape)
        out = (out.pin_memory() if pinned else out).numpy()
        loss, g = h.gradient_residual_host(a.numpy(), b.numpy(), w.numpy(), out)
        loss_d, g_d = h.gradient_residual(c.cuda(), I.cuda(), W.cuda())
        assert loss == loss_d and np.array_equal(g, g_d.cpu().numpy())
