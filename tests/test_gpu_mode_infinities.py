"""Infinite data and coefficients on handles that work in detector modes: where
the sums over channels are infinities of a sign, the results are those, and NaN
where they are NaN -- element by element those of the FP64 handle."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


def kinds(x):
    x = torch.as_tensor(x)
    return torch.isnan(x).int() + 2 * torch.isposinf(x).int() + 4 * torch.isneginf(x).int()


def same(a, b):
    b = kinds(b).cpu()
    return bool(b.any()) and torch.equal(kinds(a).cpu(), b)


# rays through a few voxels only; more than one launch of the adjoint; the caller's rows read in place (eight
# segments at l_max 8); the forward in modes (the last two; the first of them with rays through voxel centres)
CASES = [dict(n=(11, 12, 13), nj=14, nk=13, ell_max=4, n_proj=20, n_seg=8, seed=32),
         dict(n=(6, 5, 7), nj=7, nk=6, ell_max=2, n_proj=300, n_seg=5, seed=33),
         dict(n=(11, 12, 13), nj=14, nk=13, ell_max=8, n_proj=20, n_seg=8, seed=34),
         dict(n=(41, 30, 53), nj=30, nk=41, ell_max=8, n_proj=50, n_seg=16, seed=24, offsets=False),
         dict(n=(41, 30, 53), nj=31, nk=42, ell_max=6, n_proj=50, n_seg=8, seed=25)]


@pytest.mark.parametrize("kw", CASES, ids=lambda kw: f"L{kw['ell_max']}s{kw['seed']}")
@pytest.mark.parametrize("value", [float("inf"), -float("inf")])
def test_infinities_are_those_of_the_channels(kw, value):
    st = synth.small_setup(**kw)
    if not kw.get("offsets", True):
        st = dataclasses.replace(st, inner_angle=np.zeros(st.S), outer_angle=np.zeros(st.S))
    h, ref = tt.Handle(st, "f32"), tt.Handle(st, "f64")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(kw["seed"])
    c = torch.randn(st.volume_shape, device="cuda", generator=gen)
    I = torch.randn(st.data_shape, device="cuda", generator=gen)
    bad = I.clone()
    bad[2, st.nj // 2, st.nk // 2, 1] = value
    bad[4, st.nj // 2, st.nk // 3, 0] = -value
    assert same(h.adjoint(bad), ref.adjoint(bad.double()))
    for data, vol in ((bad, c), (bad, None), (I, "bad")):
        if isinstance(vol, str):
            vol = c.clone()
            vol[st.shape[0] // 2, st.shape[1] // 2, st.shape[2] // 2, 0] = value
            assert same(h.project(vol), ref.project(vol.double()))
        loss, g = h.gradient_residual(vol, data, check=False)
        loss64, g64 = ref.gradient_residual(None if vol is None else vol.double(), data.double(), check=False)
        assert same(g, g64) and not np.isfinite(loss) and not np.isfinite(loss64)   # (compensated FP32 sums: NaN)
    # finite inputs right after
    want = ref.adjoint(I.double())
    assert float((h.adjoint(I).double() - want).norm() / want.norm()) <= 1e-5


def test_the_host_entry_point_gives_them_too():
    st = synth.small_setup(**CASES[0])
    h, ref = tt.Handle(st, "f32"), tt.Handle(st, "f64")
    c = torch.randn(st.volume_shape)
    I = torch.randn(st.data_shape)
    I[2, 7, 6, 1] = float("inf")
    g = np.zeros(st.volume_shape, np.float32)
    with pytest.raises(RuntimeError):
        h.gradient_residual_host(c.numpy(), I.numpy(), None, g)
    assert same(g, ref.gradient_residual(c.double().cuda(), I.double().cuda(), check=False)[1])
