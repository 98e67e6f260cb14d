"""Edges of the regulariser kernels: volumes one plane thick, a plane short of,
at and beyond the runs of ten planes that a thread walks, rows of one voxel
and element counts that are no multiple of four.  Against the oracle: FP32 sums of at most a few rounded terms per
element (relative L2 1e-5), FP64 1e-12."""
import numpy as np
import pytest
import torch

from oracle.regularizers import l2_norm as or_l2, tv_huber as or_tv
from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("f32", 1e-5), ("f64", 1e-12)])
@pytest.mark.parametrize("n", [(1, 5, 3), (9, 1, 7), (10, 3, 1), (11, 7, 5), (21, 2, 9)])
def test_regularisers_at_run_edges(n, prec, tol):
    st = synth.small_setup(n=n, ell_max=2, n_proj=1, seed=1)
    h = tt.Handle(st, prec)
    dt = torch.float32 if prec == "f32" else torch.float64
    c = torch.as_tensor(0.1 * synth.random_volume(st, 3), dtype=dt)
    cd = c.cuda()
    ref = c.numpy().astype(np.float64)
    for (v, g), (rv, rg) in ((h.tv_huber(cd, 1e-2), or_tv(ref, 1e-2)), (h.l2_norm(cd), or_l2(ref))):
        assert abs(v - rv) <= tol * rv
        assert np.linalg.norm(g.cpu().numpy() - rg) <= tol * np.linalg.norm(rg)
    assert h.l2_norm(cd, want_grad=False)[0] == h.l2_norm(cd)[0]
