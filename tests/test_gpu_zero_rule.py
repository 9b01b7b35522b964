"""The zero rule's decisions at W = 128 and W = 256.

R = Psi - sqrt(I) Psi / |Psi|, and R = Psi where |Psi| <= 1e-5 ||p||: at the threshold R jumps by sqrt(I), so a
far-field value whose rounding reaches over it is decided by the arithmetic.  The library decides by that of its line
transforms, the same for every kernel; `golden/zero_rule_decisions.json` holds their decisions on the inputs below
(a register-resident FP32 forward model turns 7 of 99 to 102 of 605 of them).

The inputs are rational functions of the pixel, so that every machine rounds them alike.  The slices are unimodular:
dL/dconj(p) = A^H F^H R has F A dprobe = W^2 R, which gives R, and with it every decision, back from one position's
gradient."""
import json
import os

import numpy as np
import pytest
import torch

from oracle import msp_oracle as O

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "zero_rule_decisions.json")
CASES = [(128, 1), (128, 2), (128, 5), (256, 1), (256, 3)]
TOL = 1e-5


@pytest.fixture(scope="module")
def msp():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_03902_gb300 import msp
    return msp


def rel(a, b):
    a, b = np.asarray(a), np.asarray(b)
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


class Problem:
    """Slices of sharp columns under a smooth probe; every pixel of a pattern counts a hundredth of the mean amplitude."""

    def __init__(self, win, L):
        ny, nx = win + 9, win + 14
        self.gd = dict(n_slices=L, obj_ny=ny, obj_nx=nx, win=win, n_pos=1, wavelength_A=0.0698, sigma=1.5e-3, dz_A=20.0, pixel_A=0.15)
        y, x = np.arange(ny)[:, None], np.arange(nx)[None, :]
        T = []
        for l in range(L):
            t = np.zeros((ny, nx))
            for k in range(12):   # a column: a bump of width 2 pixels, at most 0.2 rad
                cy, cx = (37 * k + 11 * l) % ny, (53 * k * k + 29 * l + 7) % nx
                r2 = ((y - cy) ** 2 + (x - cx) ** 2) / 14.0
                t = t + (0.02 + 0.005 * (k % 4)) / ((1.0 + r2) * (1.0 + r2))
            T.append(((1.0 - t * t) + 2j * t) / (1.0 + t * t))
        self.T = np.array(T).astype(np.complex64)
        c = np.arange(win) - win // 2
        r2 = (c[:, None] ** 2 + c[None, :] ** 2) / (win / 10.0) ** 2
        p = (1.0 + 0.4j * r2) / ((1.0 + r2) * (1.0 + r2) * (1.0 + r2))
        self.probe = (4.0 * p).astype(np.complex64)
        self.norm = float(np.sqrt(np.sum(np.abs(self.probe.astype(np.complex128)) ** 2)))
        self.counts = np.full((win, win), np.float32((0.01 * self.norm) ** 2))

    def run(self, msp, call, windows, counts, where=1.0, **kw):
        """call(g, probe, T, pos, I) with one window and one pattern (0 or `counts`, at the pixels `where`) per position."""
        cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        g = msp.geometry(**{**self.gd, "n_pos": len(windows)}, param=msp.MSP_PARAM_TRANSMISSION)
        I = cu((self.counts * where).astype(np.float32))[None] * torch.tensor(counts, dtype=torch.float32, device="cuda")[:, None, None]
        T, p = cu(self.T), cu(self.probe)
        out = call(g, p, T, cu(np.asarray(windows, np.int32)), I.contiguous(), **kw)
        return out, T, p

    def far_field(self, wave, at):
        h = O.fresnel_propagator(self.gd["win"], self.gd["pixel_A"], self.gd["wavelength_A"], self.gd["dz_A"])
        incident, _, psi = O.position_forward(wave, self.T.astype(np.complex128), *at, h)
        return incident, psi, h

    def decisions(self, msp, at, where=1.0):
        """(bits of the values near the threshold, R, the object's gradient, which pixels these are)."""
        (loss, dT, dp), _, _ = self.run(msp, msp.loss_grad, [at], [1.0], where)
        dp = dp.cpu().numpy().astype(np.complex128)
        _, psi, _ = self.far_field(self.probe.astype(np.complex128), at)
        R = self.far_field(dp, at)[1] / self.gd["win"] ** 2
        off = np.abs(np.abs(psi) / (O.zero_threshold(self.probe.astype(np.complex128))) - 1.0)
        near = off <= 0.03 * np.sqrt(self.gd["n_slices"])
        counted = np.abs(R - psi) > 0.5 * np.sqrt(self.counts)
        return counted[near].astype(int), R, dT.cpu().numpy(), near


@pytest.mark.parametrize("win,L", CASES)
def test_values_at_the_threshold_are_decided_as_by_the_line_transforms(msp, win, L):
    q = Problem(win, L)
    with open(GOLDEN) as f:
        golden = json.load(f)
    for at in ((0, 0), (4, 9)):
        bits, R, dT, near = q.decisions(msp, at)
        want = golden[f"{win}_{L}_{at[0]}_{at[1]}"]
        assert len(bits) == len(want) and int((bits != [int(b) for b in want]).sum()) == 0
        # and the object's gradient is that of the same residual
        incident, _, h = q.far_field(q.probe.astype(np.complex128), at)
        grads, _ = O.position_backward(q.T.astype(np.complex128), *at, h, incident, O.dft2_adjoint(R), 0)
        for l, g in grads.items():
            assert rel(dT[l][at[0]:at[0] + win, at[1]:at[1] + win], g) < TOL
        # a few counts only: the pass lists these values one by one
        want = np.array([int(b) for b in want])
        for part in range(12):
            some = (np.arange(win * win).reshape(win, win) % 89 == 7 * part).astype(np.float32)
            got = q.decisions(msp, at, some)[0]
            assert (got == want * some[near]).all()


@pytest.mark.parametrize("reduce", [False, True])
@pytest.mark.parametrize("win,L", [(128, 1), (128, 5), (256, 3)])
def test_positions_decided_by_a_second_launch_beside_the_others(msp, win, L, reduce):
    """Positions of three kinds in every slot of the grid: with values at the threshold, without counts (no decision), and
    outside the object. The sums over them are the sums of single positions, in every pass; a layer and a probe step
    follow the same gradients."""
    q = Problem(win, L)
    slots = torch.cuda.get_device_properties(0).multi_processor_count // (4 if win == 256 else 1)
    S = 3 * slots + 2
    at = [(0, 0), (4, 9), (9, 14)]
    kind = (np.arange(S) * 7 // 3) % 3
    windows, counts = [at[k] for k in kind], [float(k != 1) for k in kind]
    bad = [1, 2 + slots, 4, 4 + slots, 4 + 2 * slots]
    for b in bad:
        windows[b] = (-1, 0)
    n = np.bincount(np.delete(kind, bad), minlength=3)
    one = [q.run(msp, msp.loss_grad, [at[k]], [float(k != 1)])[0] for k in range(3)]
    eT = sum(c * o[1].cpu().numpy().astype(np.complex128) for c, o in zip(n, one))
    ep = sum(c * o[2].cpu().numpy().astype(np.complex128) for c, o in zip(n, one))
    if reduce:
        msp.set_overlap_add(msp.OVERLAP_L2_REDUCE)
    try:
        (loss, dT, dp), _, _ = q.run(msp, msp.loss_grad, windows, counts)
        (only, _, _), _, _ = q.run(msp, msp.loss_grad, windows, counts, want_dV=False, want_dprobe=False)
        assert float(only) == float(loss)
        assert abs(float(loss) / sum(c * float(o[0]) for c, o in zip(n, one)) - 1) < TOL
        assert rel(dT.cpu(), eT) < TOL and rel(dp.cpu(), ep) < TOL
        if not reduce:
            (l2, dT2, dp2), _, _ = q.run(msp, msp.loss_grad, windows, counts)
            assert torch.equal(l2, loss) and torch.equal(dT2, dT) and torch.equal(dp2, dp)
        for layer in {0, L - 1, L // 2}:
            step = 1.0 / float(np.abs(eT[layer]).max())   # changes of the size of the slices, so FP32 holds them to 1e-7
            (lb, _), T, _ = q.run(msp, msp.layer_step, windows, counts, layer=layer, step=step)
            assert abs(float(lb) / float(loss) - 1) < TOL
            got = (q.T[layer].astype(np.complex128) - T.cpu().numpy()[layer]) / step
            assert rel(got, eT[layer]) < TOL
    finally:
        msp.set_overlap_add(msp.OVERLAP_FIXED_ORDER)
    step = float(np.abs(q.probe).max() / np.abs(ep).max())
    _, _, p = q.run(msp, msp.probe_step, windows, counts, step=step)
    assert rel((q.probe.astype(np.complex128) - p.cpu().numpy()) / step, ep) < TOL
