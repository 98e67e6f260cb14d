"""The mode forward's slots and the memory that others want.  They take a
sixteenth of the free memory per orientation at most: with less, the projections
go through them in more chunks, and below five slots the volume is marched
directly.  A later allocation of the library that fails gets the slots' memory.
The results stay those of a handle with all the memory it wants (the chunks bit
for bit)."""
import pytest
import torch

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu
MB = 1 << 20


def problem():
    st = synth.small_setup(n=(64, 60, 64), nj=60, nk=64, ell_max=8, n_proj=120, n_seg=8, seed=3)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    c = torch.randn(st.volume_shape, device="cuda", generator=gen)
    I = torch.randn(st.data_shape, device="cuda", generator=gen)
    return st, c, I


def fill(leave):
    """Takes device memory so that about `leave` bytes are free."""
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    return torch.empty(free - leave, dtype=torch.uint8, device="cuda") if free > leave else None


def maps(h, c):
    h.profile(True)
    h.profile_reset()
    h.project(c)
    n = h.profile_read()["pack"][1] - 1
    h.profile(False)
    return n


def test_fewer_slots_more_chunks_same_bits():
    st, c, I = problem()
    plenty = tt.Handle(st, "f32")
    want, loss, g = plenty.project(c), *plenty.gradient_residual(c, I)
    n = maps(plenty, c)
    plenty.close()
    filler = fill(4000 * MB)
    try:
        h = tt.Handle(st, "f32")
        assert maps(h, c) > n
        assert torch.equal(h.project(c), want)
        loss2, g2 = h.gradient_residual(c, I)
        assert loss2 == loss and torch.equal(g2, g)
        h.close()
    finally:
        del filler
        torch.cuda.empty_cache()


def test_no_room_for_slots():
    st, c, I = problem()
    direct = tt.Handle(st, "f32")
    direct.set_forward_kernel("l1")
    want, loss, g = direct.project(c), *direct.gradient_residual(c, I)
    direct.close()
    filler = fill(1000 * MB)
    try:
        h = tt.Handle(st, "f32")
        assert maps(h, c) == 0
        assert torch.equal(h.project(c), want)
        loss2, g2 = h.gradient_residual(c, I)
        assert loss2 == loss and torch.equal(g2, g)
        h.close()
    finally:
        del filler
        torch.cuda.empty_cache()


def test_a_solver_gets_the_slots_memory():
    """The L-BFGS state of this problem is 1.2 GB (27 vectors), the slots hold 0.8."""
    st, c, I = problem()
    h = tt.Handle(st, "f32")
    assert maps(h, c) > 0
    want = h.project(c)
    filler = fill(900 * MB)
    try:
        opt = tt.LBFGS(h, None, I, log=False)
        assert maps(h, c) == 0
        opt.step()
        got = h.project(c)
        opt.close()
    finally:
        del filler
        torch.cuda.empty_cache()
    assert float((got - want).norm()) <= 1e-6 * float(want.norm())


def test_no_room_for_the_modes():
    """60000 projections: the modes keep 0.75 GB, the rest of the handle takes 0.55.  Between the two the handle works in
    channels, as one with more modes than the mode kernels take does (two_theta = 1e-200: the same basis)."""
    st = [synth.small_setup(n=(4, 5, 6), nj=1, nk=2, ell_max=8, n_proj=60000, n_seg=16, seed=5, two_theta=t) for t in (0.0, 1e-200)]
    channels = tt.Handle(st[1], "f32")
    R = torch.randn(channels.data_shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    want = channels.adjoint(R)
    channels.close()
    room = tt.Handle(st[0], "f32")
    assert not torch.equal(room.adjoint(R), want)           # (in modes)
    room.close()
    filler = fill(950 * MB)
    try:
        h = tt.Handle(st[0], "f32")
        assert torch.equal(h.adjoint(R), want)
        h.close()
    finally:
        del filler
        torch.cuda.empty_cache()
