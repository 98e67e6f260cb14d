"""Projection and adjoint in detector modes (float handles) against the FP64
handle, whose kernels work in the K channels: the sizes at which the mode path
changes shape -- mode counts (segments below, at and above the band limit's
modes, with and without two_theta), band limits, row lengths that are no
multiple of four pixels or eight voxels, one-voxel and one-pixel problems, more
projections than a launch holds, candidate windows beyond 3 x 3 and detector
boxes that do not fit, where the handle works in channels, and the forward that
maps the volume to the modes first (which needs some work to be chosen).

Tolerance: the FP32 bound 1e-5 relative L2 of the parity tests (positions
rounded once to FP32, sums of at most N planes).
"""
import numpy as np
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu
TOL = 1e-5

CASES = [
    # band limit 2 .. 8, segments below / at / above the modes
    dict(n=(9, 7, 11), nj=8, nk=7, ell_max=2, n_proj=7, n_seg=2, seed=1),
    dict(n=(17, 9, 8), nj=9, nk=12, ell_max=2, n_proj=8, n_seg=8, seed=2),
    dict(n=(12, 13, 33), nj=17, nk=16, ell_max=4, n_proj=9, n_seg=5, seed=3),
    dict(n=(8, 4, 8), nj=8, nk=16, ell_max=4, n_proj=5, n_seg=1, seed=4),
    dict(n=(25, 10, 9), nj=33, nk=18, ell_max=4, n_proj=12, n_seg=16, seed=5),
    dict(n=(16, 12, 16), nj=15, nk=17, ell_max=6, n_proj=11, n_seg=4, seed=6),
    dict(n=(13, 9, 10), nj=16, nk=8, ell_max=6, n_proj=10, n_seg=5, seed=7),
    dict(n=(10, 11, 24), nj=12, nk=15, ell_max=6, n_proj=9, n_seg=16, seed=8),
    dict(n=(11, 8, 14), nj=13, nk=14, ell_max=8, n_proj=9, n_seg=8, seed=9),
    dict(n=(16, 16, 16), nj=16, nk=16, ell_max=8, n_proj=6, n_seg=12, seed=10),
    dict(n=(7, 9, 10), nj=10, nk=9, ell_max=8, n_proj=6, n_seg=3, seed=11),
    # a circle that is not a great circle: all modes 0 .. 2 L, and more than the path takes
    dict(n=(9, 10, 8), nj=9, nk=10, ell_max=2, n_proj=5, n_seg=8, seed=12, two_theta=0.3),
    dict(n=(9, 10, 8), nj=9, nk=10, ell_max=4, n_proj=5, n_seg=12, seed=13, two_theta=0.3),
    dict(n=(9, 10, 8), nj=9, nk=10, ell_max=6, n_proj=5, n_seg=9, seed=14, two_theta=0.2),
    dict(n=(9, 10, 8), nj=9, nk=10, ell_max=8, n_proj=5, n_seg=16, seed=15, two_theta=0.2),
    # pixels coarser and finer than voxels: other windows, then boxes that do not fit
    dict(n=(14, 12, 13), nj=9, nk=17, ell_max=4, n_proj=8, n_seg=4, seed=16, b=1.6),
    dict(n=(14, 12, 13), nj=20, nk=23, ell_max=4, n_proj=8, n_seg=6, seed=17, b=0.6),
    dict(n=(12, 12, 12), nj=40, nk=40, ell_max=8, n_proj=6, n_seg=8, seed=18, b=0.5),
    dict(n=(10, 9, 10), nj=60, nk=60, ell_max=4, n_proj=5, n_seg=6, seed=19, b=0.2),
    # enough work for the forward in modes (l_max 6 and 8, 3e6 voxels x projections)
    dict(n=(41, 30, 53), nj=31, nk=42, ell_max=6, n_proj=50, n_seg=8, seed=24),
    dict(n=(40, 33, 40), nj=40, nk=33, ell_max=6, n_proj=60, n_seg=4, seed=25),
    dict(n=(36, 50, 33), nj=50, nk=37, ell_max=6, n_proj=52, n_seg=5, seed=26, a=1.2, b=0.9),
    dict(n=(41, 30, 53), nj=24, nk=47, ell_max=8, n_proj=49, n_seg=8, seed=27),
    dict(n=(48, 31, 48), nj=33, nk=50, ell_max=8, n_proj=45, n_seg=16, seed=28),
    dict(n=(39, 47, 56), nj=48, nk=41, ell_max=8, n_proj=31, n_seg=3, seed=29),
    dict(n=(64, 57, 61), nj=21, nk=18, ell_max=8, n_proj=14, n_seg=5, seed=30, two_theta=0.1),
    # one voxel, one pixel; several launches of the adjoint
    dict(n=(1, 1, 1), nj=3, nk=2, ell_max=6, n_proj=3, n_seg=4, seed=20),
    dict(n=(5, 6, 4), nj=1, nk=1, ell_max=8, n_proj=4, n_seg=9, seed=21),
    dict(n=(6, 5, 7), nj=7, nk=6, ell_max=4, n_proj=515, n_seg=6, seed=22),
    dict(n=(6, 5, 7), nj=7, nk=6, ell_max=8, n_proj=259, n_seg=9, seed=23),
]


def rel(a, b):
    return float((a.double() - b).norm() / b.norm().clamp(min=1e-300))


@pytest.mark.parametrize("kw", CASES, ids=lambda kw: f"L{kw['ell_max']}C{kw['n_seg']}s{kw['seed']}")
def test_modes_agree_with_channels(kw):
    st = synth.small_setup(**kw)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(kw["seed"])
    c = torch.randn(st.volume_shape, device="cuda", generator=gen)
    R = torch.randn(st.data_shape, device="cuda", generator=gen)
    W = torch.rand(st.data_shape, device="cuda", generator=gen)
    h, ref = tt.Handle(st, "f32"), tt.Handle(st, "f64")
    assert rel(h.project(c), ref.project(c.double())) <= TOL
    assert rel(h.adjoint(R), ref.adjoint(R.double())) <= TOL
    for w in (None, W):
        loss, g = h.gradient_residual(c, R, w)
        loss64, g64 = ref.gradient_residual(c.double(), R.double(), None if w is None else w.double())
        assert abs(loss - loss64) <= TOL * loss64
        assert rel(g, g64) <= TOL
    # c = NULL is an all-zero volume, bit for bit
    loss0, g0 = h.gradient_residual(None, R, W)
    lossz, gz = h.gradient_residual(torch.zeros_like(c), R, W)
    assert loss0 == lossz and torch.equal(g0, gz)


def test_adjoint_reads_rows_at_any_sixteen_byte_alignment():
    """With eight segments at l_max 8 the caller's rows are the modes' rows and
    are read where they lie."""
    st = synth.small_setup(n=(9, 8, 10), nj=11, nk=9, ell_max=8, n_proj=7, n_seg=8, seed=31)
    h = tt.Handle(st, "f32")
    n = int(np.prod(st.data_shape))
    buf = torch.randn(n + 4, device="cuda")
    shifted = buf[4:].view(st.data_shape)
    assert shifted.data_ptr() % 32 == 16
    assert torch.equal(h.adjoint(shifted), h.adjoint(shifted.clone()))


@pytest.mark.parametrize("ell,seg", [(4, 8), (8, 8)])
def test_a_nonfinite_ray_reaches_only_its_voxels(ell, seg):
    """A NaN or infinite ray makes the voxels non-finite that it has a tap in,
    and no others, as in the channel kernels."""
    st = synth.small_setup(n=(11, 12, 13), nj=14, nk=13, ell_max=ell, n_proj=6, n_seg=seg, seed=32)
    h, ref = tt.Handle(st, "f32"), tt.Handle(st, "f64")
    R = torch.randn(st.data_shape, device="cuda")
    R[2, 6, 7, 1] = float("nan")
    R[4, 5, 6, 0] = float("inf")
    bad, bad64 = ~torch.isfinite(h.adjoint(R)), ~torch.isfinite(ref.adjoint(R.double()))
    assert bad.any() and not bad.all()
    assert torch.equal(bad.any(-1), bad64.any(-1))
    # the residual of such data, and finite data right after it on the same handle
    c = torch.randn(st.volume_shape, device="cuda")
    _, g = h.gradient_residual(c, R, check=False)
    _, g64 = ref.gradient_residual(c.double(), R.double(), check=False)
    assert torch.equal((~torch.isfinite(g)).any(-1), (~torch.isfinite(g64)).any(-1))
    R = torch.nan_to_num(R, nan=0.0, posinf=0.0)
    assert rel(h.gradient_residual(c, R)[1], ref.gradient_residual(c.double(), R.double())[1]) <= TOL
