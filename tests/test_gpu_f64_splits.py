"""The FP64 adjoint is the exact transpose of the FP64 projection however many CTAs
share a block's projections (one to eight, by volume and number of projections;
several launches): <A c, R> = <c, A^T R> to 1e-12 of |A c| |R|."""
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ell", [0, 2, 4, 8, 12])
@pytest.mark.parametrize("n,n_proj", [((9, 8, 10), 1), ((9, 8, 10), 3), ((16, 16, 16), 30), ((24, 23, 22), 30), ((28, 26, 27), 10),
                                      ((28, 26, 27), 120), ((36, 34, 33), 40), ((12, 11, 13), 300)])
def test_transpose(ell, n, n_proj):
    st = synth.small_setup(n=n, nj=n[1] + 2, nk=n[0] + 1, ell_max=ell, n_proj=n_proj, n_seg=6, seed=ell)
    h = tt.Handle(st, "f64")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n_proj)
    c = torch.randn(st.volume_shape, device="cuda", generator=gen, dtype=torch.float64)
    R = torch.randn(st.data_shape, device="cuda", generator=gen, dtype=torch.float64)
    Ac, AtR = h.project(c), h.adjoint(R)
    assert abs(float((Ac * R).sum() - (c * AtR).sum())) <= 1e-12 * float(Ac.norm() * R.norm())
    assert torch.equal(AtR, h.adjoint(R))
