"""The total variation's threads walk runs of ten planes on volumes that fill the
chip with them: whole runs, a last run of one plane and of all ten, by itself, in
both precisions, with and without the gradient.  Against the oracle: FP32 sums of
a few rounded terms per element (relative L2 1e-5), FP64 1e-12."""
import numpy as np
import pytest
import torch

from oracle.regularizers import tv_huber as or_tv
from paper_2504_16446_gb300 import synth, tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("f32", 1e-5), ("f64", 1e-12)])
@pytest.mark.parametrize("n", [(10, 72, 73), (11, 52, 50), (20, 52, 51), (21, 40, 44), (30, 41, 43)])
def test_total_variation_over_runs_of_ten(n, prec, tol):
    st = synth.small_setup(n=n, ell_max=4, n_proj=1, seed=1)
    blocks = -(-n[1] * n[2] * 15 // 256) * -(-n[0] // 10)
    assert blocks >= 2 * torch.cuda.get_device_properties(0).multi_processor_count   # (else the runs are shorter)
    h = tt.Handle(st, prec)
    c = torch.as_tensor(0.1 * synth.random_volume(st, 3), dtype=h.dtype)
    c[n[0] // 2:, :, : n[2] // 2] = 0                     # edges of an object, and flat ground
    v, g = h.tv_huber(c.cuda(), 1e-2)
    want, grad = or_tv(c.numpy().astype(np.float64), 1e-2)
    assert abs(v - want) <= tol * want
    assert np.linalg.norm(g.cpu().numpy() - grad) <= tol * np.linalg.norm(grad)
    assert h.tv_huber(c.cuda(), 1e-2, want_grad=False)[0] == v
