"""The network's kernels where their tile chains have edges: images narrower
than, equal to and just past a tile of 128 pixels, rows fewer than the
dilation, the smallest border (dilations 1: neighbouring image rows lie two
pixels apart), one pixel, several images and parts a CTA.  Forward layers and
parameter gradients against the CPU reference on the GPU's own BF16 inputs,
with the bounds of test_gpu_cnn.py (one BF16 step; 1e-3 of a layer's largest
gradient)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import cnn_oracle as co  # noqa: E402
from test_gpu_cnn import _acts, _net, _params  # noqa: E402

ONE = (1, 1, 1, 1, 1, 1)


@pytest.mark.parametrize("B,H,W,dil", [(1, 1, 1, ONE), (2, 5, 127, ONE), (1, 9, 128, ONE), (3, 7, 129, ONE),
                                       (2, 3, 15, (5, 2, 7, 1, 96, 3)), (1, 33, 257, (1, 1, 31, 2, 33, 1)),
                                       (5, 150, 130, (1, 3, 9, 27, 81, 1)), (40, 64, 20, ONE)])
def test_layers_and_gradients(B, H, W, dil):
    from paper_1111_0983_gb300 import cnn
    params = _params(B * H + W)
    net = _net(B, H, W, params, dil)
    rng = np.random.default_rng(W)
    g = torch.zeros(cnn.num_params(), dtype=torch.float32, device="cuda")
    out = torch.zeros((B, 2, H, W), dtype=torch.float32, device="cuda")
    for _ in range(2):   # the second pass finds the first one's buffers
        x = rng.standard_normal((B, 4, H, W)).astype(np.float32)
        dout = rng.standard_normal((B, 2, H, W)).astype(np.float32)
        net.forward(torch.from_numpy(x).cuda(), out)
        net.backward(torch.from_numpy(dout).cuda(), g)
    acts = _acts(net, B, H, W)
    P = cnn.unpack_params(cnn.pack_params(params))
    for l in range(6):
        w, b = P[l]
        z = co.conv3x3(acts[l], co.bf16_round(w), b, dil[l])
        if l < 5:
            ref, got = co.bf16_round(np.maximum(z, 0.0).astype(np.float32)), acts[l + 1]
            S = co.conv3x3(np.abs(acts[l]), np.abs(co.bf16_round(w)), np.zeros_like(b), dil[l])
            assert np.all(np.abs(got - ref) <= 2.0 ** -7 * np.maximum(np.abs(ref), np.abs(got)) + 1e-6 * S), l
        else:
            assert np.abs(out.cpu().numpy() - z).max() <= 1e-5 * np.abs(z).max()
    ref = co.CnnOracle(P, dil).backward(acts, dout.astype(np.float64))
    got = cnn.unpack_params(g.cpu().numpy())
    for l in range(6):
        for a, r in zip(got[l], ref[l]):
            assert np.abs(a - r).max() <= 1e-3 * np.abs(r).max(), l
