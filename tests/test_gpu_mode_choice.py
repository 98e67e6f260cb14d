"""Where the adjoint works in channels and where in detector modes: few projections,
many modes, volumes of more than a wave of blocks.  Seen in the bits: a two_theta
of 1e-200 gives the same basis matrix and more modes than the mode kernels take
(or pay for) at these sizes, so a handle that agrees with it bit for bit works in
channels.  Either agrees with the FP64 handle (1e-5 relative L2)."""
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu

CASES = [  # volume, l_max, segments, projections, modes?
    ((64, 60, 64), 2, 9, 39, False), ((64, 60, 64), 2, 9, 40, True),
    ((72, 70, 71), 2, 9, 15, False), ((72, 70, 71), 2, 9, 16, True), ((52, 52, 52), 2, 9, 24, False),
    ((56, 60, 64), 4, 9, 7, False), ((56, 60, 64), 4, 9, 8, True),
    ((56, 60, 64), 6, 16, 8, False), ((56, 60, 64), 6, 16, 9, True),
    ((56, 60, 64), 8, 16, 4, False), ((56, 60, 64), 8, 16, 5, True), ((56, 60, 64), 8, 16, 1, False),
    ((20, 22, 21), 6, 16, 19, False), ((20, 22, 21), 6, 16, 20, True),
    ((9, 8, 10), 8, 16, 1, False), ((9, 8, 10), 8, 16, 20, True),
]


@pytest.mark.parametrize("n,ell,n_seg,n_proj,modes", CASES)
def test_the_adjoint_by_its_projections(n, ell, n_seg, n_proj, modes):
    st = [synth.small_setup(n=n, nj=n[1] + 1, nk=n[0] - 1, ell_max=ell, n_proj=n_proj, n_seg=n_seg, seed=5, two_theta=t)
          for t in (0.0, 1e-200)]
    h, channels, ref = tt.Handle(st[0], "f32"), tt.Handle(st[1], "f32"), tt.Handle(st[0], "f64")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(6)
    R = torch.randn(st[0].data_shape, device="cuda", generator=gen)
    g = h.adjoint(R)
    assert torch.equal(g, channels.adjoint(R)) == (not modes)
    want = ref.adjoint(R.double())
    assert float((g.double() - want).norm() / want.norm()) <= 1e-5
    c = torch.randn(st[0].volume_shape, device="cuda", generator=gen)
    loss, g = h.gradient_residual(c, R)
    loss64, g64 = ref.gradient_residual(c.double(), R.double())
    assert abs(loss - loss64) <= 1e-5 * loss64 and float((g.double() - g64).norm() / g64.norm()) <= 1e-5
