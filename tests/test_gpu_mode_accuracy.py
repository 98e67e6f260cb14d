"""The forward in detector modes is as exact as the direct march on what it is
used for: volumes of a positive order-0 part and smaller higher orders, whose
projections add up whatever the map to modes rounds to one side.  Bound: 2^-22
relative L2 against the FP64 handle (a ray of N planes adds 4 N products whose
roundings are random: 2^-24 times a few; a bias of one unit in the last place
per mapped voxel alone would be 2^-23 to 2^-24 per truncated step)."""
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("ell,n_seg", [(6, 8), (6, 5), (8, 8), (8, 12), (8, 4)])
def test_objects_project_without_bias(ell, n_seg, prec):
    st = synth.small_setup(n=(64, 57, 64), nj=57, nk=64, ell_max=ell, n_proj=120, n_seg=n_seg, seed=ell)
    h, ref = tt.Handle(st, prec), tt.Handle(st, "f64")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    K = st.volume_shape[-1]
    scale = torch.cat([torch.full((2 * l + 1,), 0.5 / (1 + l), device="cuda") for l in range(0, ell + 1, 2)])
    c = torch.randn(st.volume_shape, device="cuda", generator=gen) * scale
    c[..., 0] += 2.0
    dt = {"bf16": torch.bfloat16, "f16": torch.float16}.get(prec, torch.float32)
    c = c.to(dt).float()                                   # (what the 2-byte handles store is then exact)
    want = ref.project(c.double())
    got = h.project(c).double()
    assert K == c.shape[-1] and float((got - want).norm() / want.norm()) <= 2.0 ** -22
