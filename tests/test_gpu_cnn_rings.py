"""The convolution's rings of row segments at every length the rule on shared
memory picks (it falls with the dilation), on chains several times longer and
shorter than the ring: layers and gradients against the CPU reference, with the
bounds of test_gpu_cnn_chains.py."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import test_gpu_cnn_chains as chains  # noqa: E402


@pytest.mark.parametrize("B,H,W,dil", [(1, 400, 20, (1, 8, 16, 24, 32, 1)), (1, 300, 20, (2, 40, 48, 64, 80, 2)),
                                       (2, 97, 140, (96, 96, 12, 20, 28, 96))])
def test_rings(B, H, W, dil):
    chains.test_layers_and_gradients(B, H, W, dil)
