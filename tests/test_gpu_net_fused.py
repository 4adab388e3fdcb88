"""The fused forward against the layer-by-layer one (which runs when the output
overlaps the input): the same bits, activations included, at the edges of its
8 x 32 pixel tiles."""
import ctypes

import numpy as np
import pytest

from paper_1311_3004_gb300 import fvna
from test_gpu_net import _setup, torch  # noqa: F401  (torch: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W", [(1, 1, 1), (1, 8, 32), (2, 9, 33), (3, 7, 31), (1, 70, 101),
                                   (5, 64, 64)])
def test_same_bits_as_the_layers(torch, B, H, W):  # noqa: F811
    _, _, x, net, s = _setup(torch, B=B, H=H, W=W, seed=3)
    y, h1, h2 = net.forward(x, in_scale=s, hidden=True)
    buf = x.clone()                       # output over the input
    g1, g2 = torch.empty_like(h1), torch.empty_like(h2)
    p = [ctypes.c_void_p(t.data_ptr()) for t in (buf, g1, g2)]
    rc = fvna.lib().fvna_net_forward(net._h, B, H, W, p[0], ctypes.c_float(s), p[0], p[1], p[2],
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    for a, b in ((h1, g1), (h2, g2), (y, buf)):
        assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
    net.close()
