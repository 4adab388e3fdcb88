"""The network's gradients at the edges of the training kernels' 16 x 16 pixel
tiles, against the FP64 backward on the GPU's own activations (the bound of
tests/test_gpu_net.py: FP32 sums of at most a few thousand terms)."""
import numpy as np
import pytest

from oracle import net_oracle as no
from paper_1311_3004_gb300 import fvna
from test_gpu_net import _setup, bits_to_f64, torch  # noqa: F401  (torch: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W", [(1, 1, 1), (1, 16, 16), (3, 17, 33), (2, 15, 50), (40, 31, 32)])
def test_backward_at_tile_edges(torch, B, H, W):  # noqa: F811
    p, x, xd, net, s = _setup(torch, B=B, H=H, W=W, seed=B + H + W)
    y, h1, h2 = net.forward(xd, in_scale=s, hidden=True)
    gy = np.random.default_rng(5).normal(size=x.shape).astype(np.float32)
    g = net.backward(xd, torch.from_numpy(gy).cuda(), in_scale=s).cpu().numpy()
    gd = fvna.net_params_dict(g)
    h1 = bits_to_f64(h1).transpose(0, 3, 1, 2)
    h2 = bits_to_f64(h2).transpose(0, 3, 1, 2)
    q = no.bf16
    ref = {k: 0.0 for k in gd}
    for b in range(B):
        cache = (q(x[b].astype(np.float64) * np.float32(s)), h1[b], h2[b], q(p["w1"]), q(p["w2"]),
                 q(p["w3"]))
        gb = no.backward(gy[b].astype(np.float64), cache)
        for k in ref:
            ref[k] = ref[k] + gb[k]
    for k in gd:
        err = np.max(np.abs(gd[k] - ref[k])) / (np.max(np.abs(ref[k])) + 1e-30)
        assert err < 1e-4, (k, err)
    net.close()
