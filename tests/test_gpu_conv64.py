"""The warp-specialised 64 -> 64 convolution at the edges of its strips (128
pixels, cut into 8-pixel boxes where an image is narrower) and runs of rows:
the same bits as the warp-level MMA path, which sums in the same order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 16), (2, 2, 112), (1, 3, 128), (3, 5, 144), (1, 40, 272), (2, 301, 256)])
def test_forward_and_gradients_bit_identical(gpu_lib, shape):
    import torch
    from paper_2106_01557_gb300 import lbm, surrogate
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    x = torch.randn((4,) + shape, dtype=torch.float64, device="cuda", generator=g)
    t = x + 0.1 * torch.randn(x.shape, dtype=torch.float64, device="cuda", generator=g)
    got = []
    for path in ("tcgen05", "mma"):
        s = lbm.Surrogate([0.0] * 4, [1.0] * 4, K=50, conv_path=path)
        s.set_params(surrogate.init_params(seed=3))
        out = torch.empty_like(x)
        s.forward(x, out)
        got.append((out, s.loss_grad(x, t)))
    assert torch.equal(got[0][0], got[1][0])
    assert got[0][1][0] == got[1][1][0]
    assert np.array_equal(got[0][1][1], got[1][1][1])
