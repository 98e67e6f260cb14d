"""Solves on 2-byte storage keep their bits.  Each trial volume is rounded to 11
or 8 bits, so a sum taken in another order changes a solve by whole units of the
storage: the solvers evaluate in channels, whatever a single evaluation does.

two_theta = 1e-200 gives the basis matrix of two_theta = 0 bit for bit, but twice
the detector modes (2 l_max + 1): more than the mode kernels take at l_max 6 and
8, and other ones at l_max 2 and 4.  Solves on both handles are the same bits only
when no mode kernel has part in them."""
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


def handles(ell, prec, n=(22, 19, 24), n_proj=30):
    return [tt.Handle(synth.small_setup(n=n, nj=21, nk=23, ell_max=ell, n_proj=n_proj, n_seg=16, seed=ell, two_theta=t),
                      prec) for t in (0.0, 1e-200)]


def data(h, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return 4e-3 * torch.rand(h.data_shape, device="cuda", generator=gen)


@pytest.mark.parametrize("prec", ["bf16", "f16"])
@pytest.mark.parametrize("ell", [2, 4, 6, 8])
def test_lbfgs_keeps_its_bits(ell, prec):
    a, b = handles(ell, prec)
    assert torch.equal(a.basis_matrix(), b.basis_matrix())
    I = data(a, 1)
    out = []
    for h in (a, b):
        opt = tt.LBFGS(h, None, I, log=False)
        for _ in range(3):
            opt.step()
        out.append(opt.get())
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1]) and out[0][2] == out[1][2]


@pytest.mark.parametrize("prec", ["bf16", "f16"])
@pytest.mark.parametrize("ell,n,n_proj", [(4, (22, 19, 24), 30), (8, (22, 19, 24), 30), (8, (41, 40, 44), 60)])
def test_mitra_keeps_its_bits(ell, n, n_proj, prec):
    """The last size is one whose forward goes through modes outside a solver."""
    a, b = handles(ell, prec, n, n_proj)
    I = data(a, 2)
    out = []
    for h in (a, b):
        opt = tt.MITRA(h, torch.zeros(h.volume_shape, device="cuda"), I)
        for _ in range(4):
            opt.step()
        out.append(opt.get())
    for x, y in zip(out[0], out[1]):
        assert torch.equal(x, y) if torch.is_tensor(x) else x == y


@pytest.mark.parametrize("prec", ["bf16", "f16"])
def test_ray_start_keeps_its_bits(prec):
    a, b = handles(6, prec)
    I = data(a, 3)
    u = torch.rand(a.volume_shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(4))
    loss0, g0 = a.gradient_residual(None, I)
    got = [tt.LBFGS.from_ray(h, u, g0, loss0, I, log=False) for h in (a, b)]
    assert got[0].alpha == got[1].alpha and got[0].loss == got[1].loss
    assert torch.equal(got[0].get()[1], got[1].get()[1])


@pytest.mark.parametrize("ell,n,n_proj", [(2, (22, 19, 24), 30), (4, (22, 19, 24), 30), (8, (41, 40, 44), 60)])
def test_mitra_keeps_its_bits_with_float_storage(ell, n, n_proj):
    """The preconditioner multiplies the rounding of the gradient's tap weights on voxels that few rays graze, so the
    gradient comes from the kernel that took the column sums."""
    a, b = handles(ell, "f32", n, n_proj)
    I = data(a, 5)
    out = []
    for h in (a, b):
        opt = tt.MITRA(h, torch.zeros(h.volume_shape, device="cuda"), I)
        for _ in range(4):
            opt.step()
        out.append(opt.get())
    assert all(torch.equal(x, y) for x, y in zip(out[0][:3], out[1][:3]))


@pytest.mark.parametrize("prec,unit", [("bf16", 2.0 ** -9), ("f16", 2.0 ** -12)])
@pytest.mark.parametrize("ell", [2, 4, 6, 8])
def test_lbfgs_stays_with_the_solve_in_64_bits(ell, prec, unit):
    """Rounding the trial volume to `unit` puts at most that of the projections on the residual, so that of the gradient at
    zero on the gradients (four times, for the line search's and the pairs' share), and as much of the iterate on it."""
    st = synth.small_setup(n=(22, 19, 24), nj=21, nk=23, ell_max=ell, n_proj=30, n_seg=16, seed=ell)
    h, ref = tt.Handle(st, prec), tt.Handle(st, "f64")
    I = data(h, 6)
    _, g0 = ref.gradient_residual(None, I.double())
    out = []
    for handle, d in ((h, I), (ref, I.double())):
        opt = tt.LBFGS(handle, None, d, log=False)
        for _ in range(3):
            opt.step()
        out.append(opt.get())
    (x, g, loss), (x64, g64, loss64) = out
    assert float((x.double() - x64).norm()) <= 4 * unit * float(x64.norm())
    assert float((g.double() - g64).norm()) <= 4 * unit * float(g0.norm())
