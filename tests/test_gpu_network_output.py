"""The network's ends: coefficients packed to padded bfloat16 rows, and the
last layer writing the real channels, scaled, as contiguous rows.  The same
layers run one by one through the convolution entry points (whose rows are
padded) have to give the same bits, over channel counts that fill a row of 16
or not, an odd and an even row length, and tiles that the volume cuts."""
import numpy as np
import pytest
import torch

from paper_2504_16446_gb300 import tt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k_in,k_out", [(15, 15), (16, 16), (6, 8), (1, 1), (13, 9)])
@pytest.mark.parametrize("shape", [(5, 7, 37), (1, 2, 1), (3, 9, 61), (2, 4, 30), (17, 5, 31)])
def test_network_equals_its_layers(k_in, k_out, shape):
    net = tt.WarmStartNet(k_in, k_out, seed=k_in + shape[2])
    x = torch.as_tensor(np.random.default_rng(shape[1]).normal(size=shape + (k_in,)).astype(np.float32), device="cuda")
    in_scale, out_scale = 1.75, 0.625
    got = net.forward(x, in_scale, out_scale)

    a = torch.zeros(shape + (16,), dtype=torch.bfloat16, device="cuda")
    a[..., :k_in] = (x * np.float32(1.0 / in_scale)).to(torch.bfloat16)
    lib, s, off, flat = tt.load(), torch.cuda.current_stream().cuda_stream, 0, net.weights()
    shapes = tt.WarmStartNet.layer_shapes(k_in, k_out)
    for l, shp in enumerate(shapes):
        cout, cin = shp[3:]
        w = torch.zeros((27, 32 if l < 3 else 16, 32 if l else 16), dtype=torch.bfloat16, device="cuda")
        n = int(np.prod(shp))
        w[:, :cout, :cin] = torch.as_tensor(flat[off:off + n].reshape(27, cout, cin), device="cuda").to(torch.bfloat16)
        off += n
        y = torch.empty(shape + (w.shape[1],), dtype=torch.bfloat16 if l < 3 else torch.float32, device="cuda")
        args = (*shape, w.shape[2], w.shape[1], a.data_ptr(), w.data_ptr())
        if l < 3:
            assert lib.tt_conv3d_bf16_act(*args, 1, y.data_ptr(), s) == tt.TT_OK
        else:
            assert lib.tt_conv3d_bf16(*args, 0, y.data_ptr(), s) == tt.TT_OK
        a = y
    assert torch.equal(got, np.float32(out_scale) * a[..., :k_out])
