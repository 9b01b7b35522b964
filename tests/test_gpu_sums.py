"""Sums that stand for FP64 sums hold FP64's bits: the probe gradient over the positions and the training loss.

The probe gradient's contributions are exact here.  One slice o, constant a on each position's window, and a probe that is 1
at one pixel: Psi = a everywhere, R = a (1 - sqrt(I) / |a|), and dL/dconj(p) is a^2 W^2 (1 - sqrt(I) / |a|) at that
pixel and 0 elsewhere, all of them powers of two with exact roots and transforms.  FP32 transforms of W = 64, 128 and 256 and
the precise forward models give the same numbers.  Every position has a partial sum of its own."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
FORMS = [(64, "FP32"), (128, "FP32"), (256, "FP32"), (64, "FP64_FORWARD"), (128, "DF_FORWARD")]


@pytest.fixture(scope="module")
def msp():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_03902_gb300 import msp
    return msp


def dprobe(msp, win, precision, positions):
    """positions: (a, sqrt(I) / a) each."""
    S = len(positions)
    g = msp.geometry(n_slices=1, obj_ny=win, obj_nx=win * S, win=win, n_pos=S, wavelength_A=0.0698, sigma=1.5e-3, dz_A=2.0,
                     pixel_A=0.15, param=msp.MSP_PARAM_TRANSMISSION, precision=getattr(msp, "MSP_PRECISION_" + precision))
    a = torch.tensor([p[0] for p in positions], dtype=torch.float64)
    root = a * torch.tensor([p[1] for p in positions], dtype=torch.float64)
    T = a.to(torch.complex64).repeat_interleave(win).expand(1, win, win * S).contiguous().cuda()
    I = (root * root).float()
    assert torch.equal(I.double(), root * root)
    I = I[:, None, None].expand(S, win, win).contiguous().cuda()
    probe = torch.zeros((win, win), dtype=torch.complex64, device="cuda")
    probe[0, 0] = 1.0
    pos = torch.tensor([[0, win * s] for s in range(S)], dtype=torch.int32, device="cuda")
    return msp.loss_grad(g, probe, T, pos, I)[2].cpu()


def only(win, value):
    e = torch.zeros((win, win), dtype=torch.complex64)
    e[0, 0] = value
    return e


@pytest.mark.parametrize("win,precision", FORMS)
def test_probe_gradient_keeps_the_53rd_bit_of_a_sum(msp, win, precision):
    # 1 + 2^-27 + 2^-52 - 1 - 2^-27, in units of W^2
    terms = [(1.0, 0.0), (2.0 ** -8, 1 - 2.0 ** -11), (2.0 ** -26, 0.0), (1.0, 2.0), (2.0 ** -8, 1 + 2.0 ** -11)]
    assert torch.equal(dprobe(msp, win, precision, terms), only(win, win * win * 2.0 ** -52))


@pytest.mark.parametrize("win,precision", FORMS)
def test_probe_gradient_of_a_sum_beyond_single_precision(msp, win, precision):
    # four times 2^126 and back: the sum reaches 2^128 in between
    a = 2.0 ** 63 / win
    terms = [(a, 0.0)] * 4 + [(a, 2.0)] * 4
    assert torch.equal(dprobe(msp, win, precision, terms), only(win, 0.0))
    assert torch.equal(dprobe(msp, win, precision, terms[:5]), only(win, 3 * 2.0 ** 126))
    # a partial that is not finite stays so
    assert not torch.isfinite(dprobe(msp, win, precision, [(2.0 ** 65 / win, 0.0), (1.0, 0.0)])[0, 0].real)


@pytest.mark.parametrize("win", [64, 128, 256])
def test_probe_gradient_keeps_subnormal_contributions(msp, win):
    # every position on one window, several in each slot of the grid: their own sum is a subnormal FP32 value
    S = 2 * 2 * torch.cuda.get_device_properties(0).multi_processor_count + 3
    a = 2.0 ** -70 / win   # a^2 W^2 = 2^-140
    g = msp.geometry(n_slices=1, obj_ny=win, obj_nx=win, win=win, n_pos=S, wavelength_A=0.0698, sigma=1.5e-3, dz_A=2.0,
                     pixel_A=0.15, param=msp.MSP_PARAM_TRANSMISSION)
    T = torch.full((1, win, win), a, dtype=torch.complex64, device="cuda")
    probe = torch.zeros((win, win), dtype=torch.complex64, device="cuda")
    probe[0, 0] = 1.0
    pos, I = torch.zeros((S, 2), dtype=torch.int32, device="cuda"), torch.zeros((S, win, win), device="cuda")
    assert torch.equal(msp.loss_grad(g, probe, T, pos, I)[2].cpu(), only(win, S * 2.0 ** -140))


@pytest.mark.parametrize("L", [1, 6, 8])
def test_training_loss_of_equal_squares(msp, L):
    # the value whose squares' rounding errors add up most in sums of 48 bits: 2.1e-14 at eight channels
    c = np.float32(1.4156557321548462)
    H, W = 5, 128
    s = msp.net_shape(L, H, W, scale_v=1.0, scale_g=1.0, scale_d=1.0)
    zero = torch.zeros((L, H, W), device="cuda")
    target = torch.full((L, H, W), float(c), device="cuda")
    loss, _ = msp.net_loss_grad(s, torch.zeros_like(msp.net_init(s, 1)), zero, zero, target)
    # FP64: at most 8 terms of a thread, 5 + 8 + 9 sums over its block and the blocks, two roundings of the mean
    assert abs(loss.item() / float(c) ** 2 - 1) < 32 * 2.0 ** -53
