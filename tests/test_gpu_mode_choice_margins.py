"""Where modes and channels cost about the same, the adjoint works in channels: l_max 2
with z padded by less than a quarter or less than a wave of blocks, and l_max 4 on
2-byte storage with few blocks and projections.  Seen in the bits, as a two_theta of 1e-200 keeps a handle in channels
at these sizes; either agrees with the FP64 handle (FP32 1e-5 relative L2, FP16 1e-3)."""
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu
TOL = {"f32": 1e-5, "f16": 1e-3}

CASES = [  # storage, volume, l_max, projections, modes?
    ("f32", (64, 64, 105), 2, 20, False), ("f32", (64, 64, 105), 2, 39, False), ("f32", (64, 64, 105), 2, 40, True),
    ("f32", (64, 64, 102), 2, 16, True), ("f32", (64, 64, 103), 2, 16, False), ("f16", (64, 64, 105), 2, 20, False),
    ("f32", (40, 44, 40), 2, 29, False), ("f32", (40, 44, 40), 2, 30, True), ("f16", (24, 24, 24), 2, 20, False),
    ("f16", (30, 28, 31), 4, 27, False), ("f16", (30, 28, 31), 4, 28, True), ("f32", (30, 28, 31), 4, 18, True),
    ("f16", (40, 44, 40), 4, 27, False), ("f16", (40, 44, 40), 4, 28, True), ("f16", (56, 60, 64), 4, 8, True),
]


@pytest.mark.parametrize("prec,n,ell,n_proj,modes", CASES)
def test_the_adjoint_at_the_margin(prec, n, ell, n_proj, modes):
    st = [synth.small_setup(n=n, nj=n[1] + 1, nk=n[0] - 1, ell_max=ell, n_proj=n_proj, n_seg=9, seed=5, two_theta=t)
          for t in (0.0, 1e-200)]
    h, channels, ref = tt.Handle(st[0], prec), tt.Handle(st[1], prec), tt.Handle(st[0], "f64")
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
    assert abs(loss - loss64) <= 10 * TOL[prec] * loss64
    assert float((g.double() - g64).norm() / g64.norm()) <= TOL[prec]
