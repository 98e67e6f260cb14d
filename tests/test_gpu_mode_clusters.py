"""Adjoints whose clusters split the projections, of several handles on streams
of their own: no CTA holds tensor memory while it waits for its cluster, so they
share the chip in any mix, and each gives the bits that it gives alone."""
import torch

import pytest

from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


def test_clustered_adjoints_on_streams_of_their_own():
    sets = [dict(n=(20, 19, 21), nj=22, nk=20, ell_max=4, n_proj=60, n_seg=8, seed=1),
            dict(n=(28, 26, 25), nj=27, nk=28, ell_max=2, n_proj=60, n_seg=8, seed=2),
            dict(n=(18, 20, 17), nj=20, nk=21, ell_max=8, n_proj=50, n_seg=8, seed=3),
            dict(n=(24, 22, 23), nj=25, nk=24, ell_max=6, n_proj=55, n_seg=16, seed=4)]
    work = []
    for kw in sets:
        st = synth.small_setup(**kw)
        h = tt.Handle(st, "f32")
        R = torch.randn(st.data_shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(kw["seed"]))
        work.append((h, R, h.adjoint(R), [torch.empty(st.volume_shape, device="cuda") for _ in range(8)], torch.cuda.Stream()))
    torch.cuda.synchronize()
    for t in range(8):
        for h, R, _, outs, stream in work:
            with torch.cuda.stream(stream):
                h.adjoint(R, out=outs[t])
    torch.cuda.synchronize()
    for _, _, want, outs, _ in work:
        assert all(torch.equal(o, want) for o in outs)
