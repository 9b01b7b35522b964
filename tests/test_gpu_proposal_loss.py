"""The training loss over FP32's range: the squares are summed in compensated FP32 where these hold them and in FP64
elsewhere."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 3, 8])
@pytest.mark.parametrize("scale", [1e-30, 1e-13, 1.0, 1e15, 1e18, 1e25])
def test_loss_of_a_network_that_proposes_nothing(L, scale):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_03902_gb300 import msp
    H, W = 5, 128
    s = msp.net_shape(L, H, W, scale_v=1.0, scale_g=1.0, scale_d=1.0)
    T = (scale * np.random.default_rng(L).standard_normal((L, H, W))).astype(np.float32)
    zero = torch.zeros((L, H, W), device="cuda")
    loss, _ = msp.net_loss_grad(s, torch.zeros_like(msp.net_init(s, 1)), zero, zero, torch.from_numpy(T).cuda())
    # scale_d = 1 and a proposal of 0: the differences are the targets, exactly; 640 L squares, each with 48 bits
    assert abs(loss.item() / np.mean(T.astype(np.float64) ** 2) - 1) < 1e-12
