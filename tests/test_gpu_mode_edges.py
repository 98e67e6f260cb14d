"""The adjoint in detector modes at the sizes where its kernel changes shape, with
as many projections as it takes to be chosen: mode counts of every row layout
(4, 4 + 1, 8 and 8 + 1 values), volumes that are no multiple of its 8 x 4 x 8
blocks, candidate windows beyond 3 x 3, one voxel, one pixel, a last unit of one
projection, several launches, splits of 1 to 8.  Against the FP64 handle: 1e-5
relative L2, the FP32 bound of the parity tests."""
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu
TOL = 1e-5

CASES = [
    # every row layout: R = 2, 3, 4, 5 | 5, 6, 8, 9
    dict(n=(9, 7, 11), nj=8, nk=7, ell_max=2, n_proj=25, n_seg=2, seed=1),
    dict(n=(17, 9, 8), nj=9, nk=12, ell_max=2, n_proj=21, n_seg=8, seed=2),
    dict(n=(8, 4, 8), nj=8, nk=16, ell_max=4, n_proj=21, n_seg=1, seed=4),
    dict(n=(25, 10, 9), nj=33, nk=18, ell_max=4, n_proj=23, n_seg=4, seed=5),
    dict(n=(12, 13, 33), nj=17, nk=16, ell_max=4, n_proj=23, n_seg=5, seed=3),
    dict(n=(13, 9, 10), nj=16, nk=8, ell_max=6, n_proj=24, n_seg=5, seed=7),
    dict(n=(10, 11, 24), nj=12, nk=15, ell_max=6, n_proj=21, n_seg=16, seed=8),
    dict(n=(11, 8, 14), nj=13, nk=14, ell_max=8, n_proj=25, n_seg=8, seed=9),
    dict(n=(16, 16, 16), nj=16, nk=16, ell_max=8, n_proj=20, n_seg=12, seed=10),
    dict(n=(7, 9, 10), nj=10, nk=9, ell_max=8, n_proj=22, n_seg=3, seed=11),
    # all modes 0 .. 2 L of a circle that is no great circle
    dict(n=(9, 10, 8), nj=9, nk=10, ell_max=2, n_proj=24, n_seg=8, seed=12, two_theta=0.3),
    dict(n=(9, 10, 8), nj=9, nk=10, ell_max=4, n_proj=21, n_seg=12, seed=13, two_theta=0.3),
    dict(n=(9, 10, 8), nj=9, nk=10, ell_max=6, n_proj=21, n_seg=9, seed=14, two_theta=0.2),
    # pixels coarser and finer than voxels
    dict(n=(14, 12, 13), nj=9, nk=17, ell_max=4, n_proj=24, n_seg=4, seed=16, b=1.6),
    dict(n=(14, 12, 13), nj=20, nk=23, ell_max=4, n_proj=24, n_seg=6, seed=17, b=0.6),
    dict(n=(14, 12, 13), nj=20, nk=23, ell_max=2, n_proj=24, n_seg=6, seed=18, b=0.6),
    # one voxel, one pixel, several launches (256 projections each), the last of them short
    dict(n=(1, 1, 1), nj=3, nk=2, ell_max=6, n_proj=21, n_seg=4, seed=20),
    dict(n=(5, 6, 4), nj=1, nk=1, ell_max=8, n_proj=20, n_seg=9, seed=21),
    dict(n=(6, 5, 7), nj=7, nk=6, ell_max=2, n_proj=513, n_seg=6, seed=22),
    # volumes whose clusters split by 8, 4, 2 and 1
    dict(n=(16, 12, 16), nj=15, nk=17, ell_max=4, n_proj=100, n_seg=5, seed=24),
    dict(n=(33, 26, 30), nj=30, nk=31, ell_max=6, n_proj=60, n_seg=8, seed=25),
    dict(n=(41, 42, 39), nj=40, nk=41, ell_max=8, n_proj=40, n_seg=8, seed=26),
    dict(n=(57, 66, 49), nj=50, nk=51, ell_max=4, n_proj=30, n_seg=8, seed=27),
    dict(n=(70, 66, 83), nj=55, nk=61, ell_max=2, n_proj=45, n_seg=8, seed=28),
]


@pytest.mark.parametrize("kw", CASES, ids=lambda kw: f"L{kw['ell_max']}C{kw['n_seg']}s{kw['seed']}")
@pytest.mark.parametrize("prec", ["f32", "bf16"])
def test_modes_at_their_edges(kw, prec):
    st = synth.small_setup(**kw)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(kw["seed"])
    R = torch.randn(st.data_shape, device="cuda", generator=gen)
    W = torch.rand(st.data_shape, device="cuda", generator=gen)
    h, ref = tt.Handle(st, prec), tt.Handle(st, "f64")
    want = ref.adjoint(R.double())
    assert float((h.adjoint(R).double() - want).norm() / want.norm()) <= TOL
    # at zero, where 2-byte storage rounds nothing
    loss, g = h.gradient_residual(None, R, W)
    loss64, g64 = ref.gradient_residual(None, R.double(), W.double())
    assert abs(loss - loss64) <= TOL * loss64
    assert float((g.double() - g64).norm() / g64.norm()) <= TOL
    if prec == "f32":
        c = torch.randn(st.volume_shape, device="cuda", generator=gen)
        loss, g = h.gradient_residual(c, R, W)
        loss64, g64 = ref.gradient_residual(c.double(), R.double(), W.double())
        assert abs(loss - loss64) <= TOL * loss64
        assert float((g.double() - g64).norm() / g64.norm()) <= TOL


@pytest.mark.parametrize("ell,seg,n,n_proj", [(4, 8, (11, 12, 13), 20), (8, 8, (11, 12, 13), 21), (2, 8, (11, 12, 13), 20),
                                             (6, 8, (41, 30, 53), 50), (8, 16, (41, 30, 53), 50)])
def test_a_nonfinite_ray_reaches_only_its_voxels(ell, seg, n, n_proj):
    """The adjoint adds no zero times NaN to voxels that only list the ray; an evaluation, whose loss is then not
    finite, is taken again in channels (the last two after a forward in modes)."""
    st = synth.small_setup(n=n, nj=n[1] + 2, nk=n[0] + 1, ell_max=ell, n_proj=n_proj, n_seg=seg, seed=32)
    h, ref = tt.Handle(st, "f32"), tt.Handle(st, "f64")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    R = torch.randn(st.data_shape, device="cuda", generator=gen)
    c = torch.randn(st.volume_shape, device="cuda", generator=gen)
    bad = R.clone()
    bad[2, n[1] // 2, n[0] // 2, 1] = float("nan")
    nan, nan64 = torch.isnan(h.adjoint(bad)), torch.isnan(ref.adjoint(bad.double()))
    assert nan64.any() and not nan64.all() and torch.equal(nan, nan64)
    _, g = h.gradient_residual(c, bad, check=False)
    _, g64 = ref.gradient_residual(c.double(), bad.double(), check=False)
    assert torch.equal(torch.isnan(g), torch.isnan(g64))
    want = ref.gradient_residual(c.double(), R.double())[1]
    assert float((h.gradient_residual(c, R)[1].double() - want).norm() / want.norm()) <= TOL
