"""Detectors that the volume's shadow covers little of take the direct march with
another number of resident CTAs: the same rays give the same bits as on a detector
that fits the volume, and the rest is zero.  Both agree with the FP64 handle
(1e-5 relative L2; 2-byte storage: as in the precision tests)."""
import dataclasses

import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu
TOL = {"f32": 1e-5, "bf16": 5e-3, "f16": 1e-3}


@pytest.mark.parametrize("prec,ell", [("f32", 6), ("bf16", 4), ("f16", 4), ("f32", 10), ("f32", 12), ("bf16", 6), ("f16", 10),
                                      ("bf16", 12)])
@pytest.mark.parametrize("n_seg", [5, 8])
def test_wide_detectors(prec, ell, n_seg):
    near = synth.small_setup(n=(20, 17, 19), nj=20, nk=24, ell_max=ell, n_proj=7, n_seg=n_seg, seed=ell)
    far = dataclasses.replace(near, nj=20 + 2 * 31, nk=24 + 2 * 40)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    c = torch.randn(near.volume_shape, device="cuda", generator=gen)
    a, b, ref = tt.Handle(near, prec), tt.Handle(far, prec), tt.Handle(far, "f64")
    want, got = ref.project(c.double()), b.project(c)
    assert float((got.double() - want).norm() / want.norm()) <= TOL[prec]
    assert torch.equal(got[:, 31:-31, 40:-40], a.project(c))
    I = torch.randn(far.data_shape, device="cuda", generator=gen)
    loss, g = b.gradient_residual(c, I)
    loss64, g64 = ref.gradient_residual(c.double(), I.double())
    assert abs(loss - loss64) <= 10 * TOL[prec] * loss64
    assert float((g.double() - g64).norm() / g64.norm()) <= TOL[prec]
