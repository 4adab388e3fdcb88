"""Many images that fill little of their 8 x 32 pixel tiles: a forward takes no
longer than the layers one by one (which run when the output overlaps the
input), and gives their bits.  Shortest of fifteen runs each, in turn; the
fused kernel took 1.11 to 1.14 times as long here, runs scatter by a percent or two."""
import ctypes
import time

import numpy as np
import pytest

from paper_1311_3004_gb300 import fvna
from test_gpu_net import _setup, torch  # noqa: F401  (torch: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W", [(60000, 1, 1), (8192, 9, 33)])
def test_no_slower_than_the_layers(torch, B, H, W):  # noqa: F811
    _, _, _, net, s = _setup(torch, B=1, H=8, W=8, seed=3)
    x = torch.randn((B, 3, H, W), device="cuda", dtype=torch.float32)
    y, buf = torch.empty_like(x), torch.empty_like(x)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def forward(src, dst):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        rc = fvna.lib().fvna_net_forward(net._h, B, H, W, ctypes.c_void_p(src.data_ptr()),
                                         ctypes.c_float(s), ctypes.c_void_p(dst.data_ptr()), None,
                                         None, stream)
        assert rc == 0
        return time.perf_counter() - t0

    apart = over = 1e9
    for _ in range(15):
        apart = min(apart, forward(x, y))
        buf.copy_(x)
        over = min(over, forward(buf, buf))
    assert np.array_equal(y.cpu().numpy(), buf.cpu().numpy())
    assert apart <= 1.07 * over, (apart, over)
    net.close()
