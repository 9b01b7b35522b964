"""The measured calls of the library: what a program that uses it has it compute.

A case is a dict of plain values.  `kind` names the public entry point:

  forward      msp.forward: the intensities of a specimen (simulation, checking a proposal)
  grad         msp.loss_grad: the loss, dV of every slice and dprobe
  autograd     msp.multislice_loss and its backward: the same through torch.autograd
  layer        msp.layer_step: one step of Algorithm 1 on one slice
  reconstruct  msp.reconstruct: sweeps of Algorithm 1 with probe steps, a whole call
  smd          msp.smd_matrix_step and msp.smd_decompose: one iteration of Algorithm 2
  train        msp.net_train_step: one Adam step of the proposal network

The listed sizes are those of `workloads/synth.py` (c1 to c5 and the GaAs setting of Algorithm 2),
with odd object sides and odd position counts where nothing fixes them.

Inputs are drawn on the device from the seed by plain torch, never by the library: thick slices of
heavy columns (0.3 to 0.7 rad at the site, the columns of the GaAs setting in 2 nm slices), patterns
of the true specimen and probe with counting noise, and the state of the first sweeps of a
reconstruction: site amplitudes still far below the true ones and a probe guess 20 A off in defocus
and a third too low in beam current (a pattern sum is known to the detector gain only).

The multislice calls in FP32 and the network sum FP32 terms into an FP64 scalar (the loss, the step
size).  Only its leading digits mean anything and programs log it in single precision, so `run`
returns it that way; the precise form's loss is FP64 throughout and is returned as it is.
"""
import math

import torch

from paper_2205_03902_gb300 import msp

LAMBDA_A = 0.06979081578546553      # electron wavelength and interaction constant at 30 kV
SIGMA = 0.001543269908404932        # (workloads/physics.py)
SMD_LAMBDA_A = 0.025079340450548007  # wavelength at 200 kV
DZ_A = 20.0
LATTICE_A, SITE_A = 3.9, 0.3
AMPLITUDE = (200.0, 450.0)          # V angstrom at a site
DOSE = 1e6                          # counts per pattern
ZERO_TAU = 1e-5                     # a far-field value at or below tau ||p|| counts as zero (include/msp.h)


def _dev():
    return torch.device("cuda", torch.cuda.current_device()) if torch.cuda.is_available() else torch.device("cpu")


# ---------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------
def _scan(kind, win, n_slices, scan_ny, scan_nx, step_px, extra_y=0, extra_x=0, **more):
    """A raster of scan_ny x scan_nx windows; the object is the raster's extent and `extra` pixels."""
    return dict(kind=kind, win=win, n_slices=n_slices, scan_ny=scan_ny, scan_nx=scan_nx, step_px=step_px,
                obj_ny=(scan_ny - 1) * step_px + win + extra_y, obj_nx=(scan_nx - 1) * step_px + win + extra_x,
                **{**dict(param="potential", precision="fp32"), **more})


def listed():
    return [
        # the smallest call: a W = 64 pattern set simulated from two slices (c1's size)
        dict(_scan("forward", 64, 2, 8, 8, 4, 4, 4), name="forward_w64_s64"),
        # the plain method at c1's size with probe estimation: short passes in a long chain
        dict(_scan("reconstruct", 64, 2, 8, 8, 4, 4, 4, sweeps=3, probe_steps=1), name="reconstruct_w64_s64"),
        # a 64-pixel detector over a fine odd raster, the ordinary size of a fast 4D-STEM camera
        dict(_scan("grad", 64, 5, 47, 45, 5, 3, 6), name="grad_w64_s2115"),
        # c2: the forward model alone (simulating data, judging a proposal)
        dict(_scan("forward", 128, 4, 32, 32, 8, 8, 8), name="forward_w128_s1024"),
        # c2: the headline loss-and-gradient step
        dict(_scan("grad", 128, 4, 32, 32, 8, 8, 8), name="grad_w128_s1024"),
        # c2: the unit of Algorithm 1
        dict(_scan("layer", 128, 4, 32, 32, 8, 8, 8, layer=2), name="layer_w128_s1024"),
        # c3: eight slices, four times the positions
        dict(_scan("grad", 128, 8, 64, 64, 4, 4, 4), name="grad_w128_s4096"),
        # the paper's own unknowns (complex slices) on a ragged scan of an odd object
        dict(_scan("grad", 128, 3, 21, 16, 9, 5, 10, param="transmission"), name="transmission_w128_s336"),
        # precise gradients near a fit: the double-float forward on a 13 x 13 sub-scan
        dict(_scan("grad", 128, 4, 13, 13, 8, 9, 0, precision="df"), name="precise_w128_s169"),
        # c4: sixteen slices, W = 256, through torch.autograd; the largest
        dict(_scan("autograd", 256, 16, 48, 48, 8, 8, 8), name="autograd_w256_s2304"),
        # Algorithm 2 in Table 1's GaAs setting: every cyclic shift of a 40 x 40 probe, three slices
        dict(kind="smd", name="smd_n40_s1600", n=40, n_slices=3, n_pos=1600),
        # training the proposal network at c5's size
        dict(kind="train", name="train_l8_384", n_slices=8, height=384, width=384),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["forward", "grad", "grad", "grad", "layer", "autograd", "reconstruct", "precise", "transmission",
                       "smd", "train"])
    if kind == "smd":
        n = rng.choice([16, 24, 32, 40, 48])
        return dict(kind="smd", n=n, n_slices=rng.randint(1, 4), n_pos=spread(max(16, n), min(n * n, 1800)))
    if kind == "train":
        return dict(kind="train", n_slices=rng.randint(1, 8), height=spread(96, 900), width=128 * rng.randint(1, 6))
    win = rng.choice([64, 128, 128, 256])
    # positions up to c3's 4096, fewer where a position costs more; a c4 pass is the dearest
    most = {64: 4096, 128: 4096, 256: 1500}[win]
    slices = rng.randint(1, {64: 12, 128: 10, 256: 12}[win])
    if kind == "reconstruct":
        most, slices = {64: 800, 128: 300, 256: 120}[win], min(slices, 4)
    if kind == "precise":
        win, most, slices = min(win, 128), 350, min(slices, 6)
    s = spread(12, most)
    ny = max(2, int(round(math.sqrt(s) * rng.uniform(0.7, 1.4))))
    nx = max(2, s // ny)
    step = rng.randint(2, 11)
    more = dict(extra_y=rng.randint(0, 33), extra_x=rng.randint(0, 33))
    if kind == "reconstruct":
        return _scan("reconstruct", win, slices, ny, nx, step, **more, sweeps=rng.randint(1, 2), probe_steps=rng.randint(0, 1))
    if kind == "layer":
        return _scan("layer", win, slices, ny, nx, step, **more, layer=rng.randrange(slices))
    if kind == "precise":
        return _scan("grad", win, slices, ny, nx, step, **more, precision="df")
    if kind == "transmission":
        return _scan("grad", win, slices, ny, nx, step, **more, param="transmission")
    return _scan(kind, win, slices, ny, nx, step, **more)


# ---------------------------------------------------------------------------------------------
# inputs (plain torch)
# ---------------------------------------------------------------------------------------------
def _pixel(case):
    return {64: 0.2, 128: 0.15, 256: 0.1}[case["win"]]


def _gen(seed, dev):
    return torch.Generator(device=dev).manual_seed(int(seed) * 7919 + 17)


def _uniform(shape, lo, hi, gen):
    return torch.rand(shape, generator=gen, device=gen.device, dtype=torch.float32) * (hi - lo) + lo


def _columns(L, ny, nx, px, gen):
    """(site amplitudes, row and column profiles) of every slice: a square lattice of Gaussian columns
    with a random offset and 30 % vacancies; the slice is rows^T amplitudes columns."""
    dev = gen.device
    my, mx = int(ny * px / LATTICE_A) + 2, int(nx * px / LATTICE_A) + 2
    off = _uniform((L, 2), 0.0, LATTICE_A, gen)
    amp = _uniform((L, my, mx), *AMPLITUDE, gen) * (torch.rand((L, my, mx), generator=gen, device=dev) >= 0.3)

    def profile(m, n, o):
        at = (torch.arange(m, device=dev, dtype=torch.float32) - 1) * LATTICE_A + o[:, None]
        x = torch.arange(n, device=dev, dtype=torch.float32) * px
        return torch.exp(-((x[None, None, :] - at[:, :, None]) ** 2) / (2 * SITE_A ** 2))

    return amp, profile(my, ny, off[:, 0]), profile(mx, nx, off[:, 1])


def _slices(amp, rows, cols):
    return (rows.transpose(1, 2) @ amp @ cols).contiguous()


def _frequencies(w, px, dev):
    return torch.fft.fftfreq(w, d=px, dtype=torch.float64).to(dev)


def _probe(w, px, lam, mrad, defocus, norm2, dev):
    q = _frequencies(w, px, dev)
    q2 = q[:, None] ** 2 + q[None, :] ** 2
    spec = torch.polar((q2 <= (mrad * 1e-3 / lam) ** 2).double(), -math.pi * lam * defocus * q2)
    p = torch.fft.fftshift(torch.fft.ifft2(spec))
    return p * math.sqrt(norm2 / float(p.abs().square().sum()))


def _fresnel(w, px, lam, dz, dev):
    q = _frequencies(w, px, dev)
    q2 = q[:, None] ** 2 + q[None, :] ** 2
    return torch.polar(torch.ones_like(q2), -math.pi * dz * lam * q2)


def _positions(case, dev):
    y = torch.arange(case["scan_ny"], device=dev) * case["step_px"] + (case["obj_ny"] - case["win"] - (case["scan_ny"] - 1) * case["step_px"]) // 2
    x = torch.arange(case["scan_nx"], device=dev) * case["step_px"] + (case["obj_nx"] - case["win"] - (case["scan_nx"] - 1) * case["step_px"]) // 2
    yy, xx = torch.meshgrid(y, x, indexing="ij")
    return torch.stack([yy.reshape(-1), xx.reshape(-1)], dim=1).to(torch.int32).contiguous()


def _windows(X, pos, w):
    """[B][w][w] windows of one slice."""
    r = torch.arange(w, device=X.device)
    y, x = pos[:, 0].long(), pos[:, 1].long()
    return X[(y[:, None] + r)[:, :, None], (x[:, None] + r)[:, None, :]]


def _batch(w):
    return max(1, (1 << 22) // (w * w))


def _inputs(case, seed):
    dev = _dev()
    gen = _gen(seed, dev)
    w, L, px = case["win"], case["n_slices"], _pixel(case)
    pos = _positions(case, dev)
    amp, rows, cols = _columns(L, case["obj_ny"], case["obj_nx"], px, gen)
    V_true = _slices(amp, rows, cols)
    V = _slices(amp * _uniform(tuple(amp.shape), 0.0, 0.5, gen), rows, cols)   # the estimate so far
    probe_true = _probe(w, px, LAMBDA_A, 30.0, 100.0, DOSE / w ** 2, dev).to(torch.complex64)
    probe = _probe(w, px, LAMBDA_A, 30.0, 120.0, 0.65 * DOSE / w ** 2, dev).to(torch.complex64)
    h = _fresnel(w, px, LAMBDA_A, DZ_A, dev).to(torch.complex64)
    I = torch.empty((len(pos), w, w), dtype=torch.float32, device=dev)
    X = [torch.polar(torch.ones_like(v), SIGMA * v) for v in V_true]
    for b in range(0, len(pos), _batch(w)):
        ps = pos[b:b + _batch(w)]
        psi = probe_true.expand(len(ps), w, w)
        for l in range(L):
            psi = psi * _windows(X[l], ps, w)
            if l < L - 1:
                psi = torch.fft.ifft2(torch.fft.fft2(psi) * h)
        I[b:b + len(ps)] = torch.poisson(torch.fft.fft2(psi).abs().square(), generator=gen)
    if case["param"] == "transmission":   # the estimate as complex slices, slightly absorbing
        V = torch.polar(1.0 - 0.1 * _uniform(tuple(V.shape), 0.0, 1.0, gen), SIGMA * V)
    return dict(probe=probe, V=V, pos=pos, I=I)


def _smd_inputs(case, seed):
    dev = _dev()
    gen = _gen(seed, dev)
    n, M, S, px = case["n"], case["n_slices"], case["n_pos"], 2 * 5.6533 / 40
    shifts = torch.randperm(n * n, generator=gen, device=dev)[:S].sort().values
    shifts = torch.stack([shifts // n, shifts % n], dim=1).to(torch.int32).contiguous()
    probe = _probe(n, px, SMD_LAMBDA_A, 32.0, 0.0, 1.0, dev)
    o = torch.polar(torch.ones((M, n, n), device=dev, dtype=torch.float64),
                    0.3 * torch.randn((M, n, n), generator=gen, device=dev, dtype=torch.float64))
    h = _fresnel(n, px, SMD_LAMBDA_A, 20.0, dev)
    ps = torch.stack([torch.roll(probe, (int(a), int(b)), (0, 1)) for a, b in shifts.tolist()])
    for m in range(M):
        ps = ps * o[m]
        if m < M - 1:
            ps = torch.fft.ifft2(torch.fft.fft2(ps) * h)
    I = torch.fft.fft2(ps).abs().square()
    o0 = o.angle() * 0.5 + 0.1 * torch.randn((M, n, n), generator=gen, device=dev, dtype=torch.float64)
    o0 = torch.polar(torch.full_like(o0, 1.0 / n), o0)   # unit Frobenius norm, as Algorithm 2 keeps them
    A0 = _transfer(o0, h) * float(n) ** M * 0.9
    return dict(probe=probe.to(torch.complex64), shifts=shifts, I=I.float(), o=o0.to(torch.complex64),
                lam=torch.full((1,), 0.9 * float(n) ** M, dtype=torch.float64, device=dev), A=A0.to(torch.complex64))


def _transfer(o, h):
    """Row j: the exit wave of an impulse at pixel j, [n^2][n^2]."""
    n = o.shape[-1]
    e = torch.eye(n * n, dtype=o.dtype, device=o.device).reshape(n * n, n, n)
    for m in range(len(o)):
        e = e * o[m]
        if m < len(o) - 1:
            e = torch.fft.ifft2(torch.fft.fft2(e) * h)
    return e.reshape(n * n, n * n)


def _net_layout(L):
    ch = [2 * L, 64, 64, 64, 64, 64, L]
    out, off = [], 0
    for i in range(6):
        out.append((ch[i], ch[i + 1], off, off + ch[i + 1] * 9 * ch[i]))
        off += ch[i + 1] * (9 * ch[i] + 1)
    return out, off


def _net_inputs(case, seed):
    """Mid-training: trained-size weights and Adam moments, potentials, gradients and a target."""
    dev = _dev()
    gen = _gen(seed, dev)
    L, H, W = case["n_slices"], case["height"], case["width"]
    lay, n = _net_layout(L)
    p = torch.zeros(n, device=dev)
    for ci, co, a, b in lay:
        p[a:b] = _uniform((b - a,), -1.0, 1.0, gen) * math.sqrt(6.0 / (9 * ci + 9 * co))
        p[b:b + co] = _uniform((co,), -0.05, 0.05, gen)
    V = _slices(*_columns(L, H, W, 0.15, gen)) / 400.0
    G = 0.3 * torch.randn((L, H, W), generator=gen, device=dev) * (0.2 + V)
    target = 0.5 * V + 0.05 * torch.randn((L, H, W), generator=gen, device=dev)
    return dict(p=p, m=1e-4 * torch.randn(n, generator=gen, device=dev),
                v=1e-7 * (0.5 + torch.rand(n, generator=gen, device=dev)), V=V, G=G, target=target)


# ---------------------------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------------------------
def _geometry(case):
    return msp.geometry(
        n_slices=case["n_slices"], obj_ny=case["obj_ny"], obj_nx=case["obj_nx"], win=case["win"],
        n_pos=case["scan_ny"] * case["scan_nx"], wavelength_A=LAMBDA_A, sigma=SIGMA, dz_A=DZ_A, pixel_A=_pixel(case),
        param=msp.MSP_PARAM_TRANSMISSION if case["param"] == "transmission" else msp.MSP_PARAM_POTENTIAL,
        precision=msp.MSP_PRECISION_DF_FORWARD if case["precision"] == "df" else msp.MSP_PRECISION_FP32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "smd":
        s = _smd_inputs(case, seed)
        s["g"] = msp.smd_geometry(n=case["n"], n_slices=case["n_slices"], n_pos=case["n_pos"], wavelength_A=SMD_LAMBDA_A,
                                  dz_A=20.0, pixel_A=2 * 5.6533 / 40)
        s["ws"] = msp.smd_make_workspace(s["g"])
    elif kind == "train":
        s = _net_inputs(case, seed)
        s["g"] = msp.net_shape(case["n_slices"], case["height"], case["width"], 1.0, 1.0, 0.5)
        s["ws"] = msp.net_make_workspace(s["g"])
        s["step"] = 100
    else:
        s = _inputs(case, seed)
        s["g"] = _geometry(case)
        s["ws"] = msp.make_workspace(s["g"])
        if kind == "autograd":
            s["V"].requires_grad_(True)
            s["probe"].requires_grad_(True)
        if kind == "reconstruct":
            s["plan"] = msp.plan(case["sweeps"], probe_steps=case["probe_steps"])
    s["case"] = dict(case)
    return s


def run(s):
    case, g, ws = s["case"], s["g"], s["ws"]
    kind = case["kind"]
    if kind == "forward":
        return {"I": msp.forward(g, s["probe"], s["V"], s["pos"], ws=ws)}
    if kind == "grad":
        loss, dV, dprobe = msp.loss_grad(g, s["probe"], s["V"], s["pos"], s["I"], ws=ws)
        return {"loss": loss if case["precision"] == "df" else loss.float(), "dV": dV, "dprobe": dprobe}
    if kind == "autograd":
        loss = msp.multislice_loss(g, s["V"], s["probe"], s["pos"], s["I"], ws=ws)
        dV, dprobe = torch.autograd.grad(loss, (s["V"], s["probe"]))
        return {"loss": loss.detach().float(), "dV": dV, "dprobe": dprobe}
    if kind == "layer":
        loss, mu = msp.layer_step(g, s["probe"], s["V"], s["pos"], s["I"], layer=case["layer"], ws=ws)
        return {"loss": loss.float(), "mu": mu.float(), "V": s["V"]}
    if kind == "reconstruct":
        history = msp.reconstruct(g, s["plan"], s["probe"], s["V"], s["pos"], s["I"], ws=ws)
        return {"history": history.float(), "V": s["V"], "probe": s["probe"]}
    if kind == "smd":
        objective, mu = msp.smd_matrix_step(g, s["A"], s["probe"], s["shifts"], s["I"], ws=ws)
        before = msp.smd_decompose(g, s["A"], s["o"], s["lam"], ws=ws)
        return {"objective": objective.float(), "mu": mu.float(), "before": before.float(), "A": s["A"], "o": s["o"],
                "lam": s["lam"].float()}
    loss = msp.net_train_step(g, s["p"], s["m"], s["v"], s["step"], 1e-4, s["V"], s["G"], s["target"], ws=ws)
    s["step"] += 1
    return {"loss": loss.float(), "p": s["p"], "m": s["m"], "v": s["v"]}


def work(case):
    kind = case["kind"]
    if kind == "smd":
        n2, S, M = case["n"] ** 2, case["n_pos"], case["n_slices"]
        image = 2 * 5 * n2 * math.log2(n2)
        # two complex contractions; per column of A about 4 (M - 1) image transforms; two per pattern
        flops = 2 * 8 * n2 * n2 * S + image * (S + n2 * 4 * max(1, M - 1))
        return {"bytes": 2 * 8 * n2 * n2 + 4 * S * n2 + 2 * 8 * M * n2, "flops": flops}
    if kind == "train":
        lay, n = _net_layout(case["n_slices"])
        pix = case["height"] * case["width"]
        macs = sum(ci * 9 * co for ci, co, _, _ in lay)
        first = lay[0][0] * 9 * lay[0][1]
        return {"bytes": 3 * 4 * case["n_slices"] * pix + 2 * 3 * 4 * n, "flops": 2 * pix * (3 * macs - first)}
    w2, S, L = case["win"] ** 2, case["scan_ny"] * case["scan_nx"], case["n_slices"]
    plane = case["obj_ny"] * case["obj_nx"] * (8 if case["param"] == "transmission" else 4)
    image = 5 * w2 * math.log2(w2)
    way = (2 * L - 1) * image * S
    back = {"grad": way, "autograd": way}.get(kind, 0)
    if kind == "forward":
        return {"bytes": 8 * w2 + L * plane + 4 * S * w2, "flops": way}
    if kind == "layer":
        return {"bytes": 8 * w2 + (L + 1) * plane + 4 * S * w2, "flops": way + (2 * (L - 1 - case["layer"]) + 1) * image * S}
    if kind == "reconstruct":
        sweep = sum(way + (2 * (L - 1 - l) + 1) * image * S for l in range(L)) + case["probe_steps"] * 2 * way
        # each step reads the patterns: every one depends on the step before
        steps = case["sweeps"] * (L + case["probe_steps"]) + 1
        return {"bytes": steps * (8 * w2 + (L + 1) * plane + 4 * S * w2), "flops": case["sweeps"] * sweep + way}
    return {"bytes": 2 * 8 * w2 + 2 * L * plane + 4 * S * w2, "flops": way + back}


# ---------------------------------------------------------------------------------------------
# the same results in 64 bits, by plain torch
# ---------------------------------------------------------------------------------------------
def _pass(case, probe, X, pos, I, lowest=0, h=None):
    """(patterns or None, loss, dX, dprobe, illumination of slice `lowest`): the multislice recursion,
    the amplitude residual and the adjoint (Sec. 2.1, 3.2, 3.3), every position, complex128."""
    w, L, dev = case["win"], len(X), probe.device
    h = _fresnel(w, _pixel(case), LAMBDA_A, DZ_A, dev)
    thr = ZERO_TAU * float(probe.abs().square().sum().sqrt())
    plane = X[0].numel()
    dX = torch.zeros((L, plane), dtype=torch.complex128, device=dev)
    illum = torch.zeros(plane, dtype=torch.float64, device=dev)
    dprobe = torch.zeros((w, w), dtype=torch.complex128, device=dev)
    loss = torch.zeros((), dtype=torch.float64, device=dev)
    pats = None if I is not None else torch.empty((len(pos), w, w), dtype=torch.float64, device=dev)
    r = torch.arange(w, device=dev)
    nx = X[0].shape[1]
    B = max(1, _batch(w) // 4)
    for b in range(0, len(pos), B):
        ps = pos[b:b + B]
        psi, into = probe.expand(len(ps), w, w), []
        for l in range(L):
            into.append(psi)
            psi = psi * _windows(X[l], ps, w)
            if l < L - 1:
                psi = torch.fft.ifft2(torch.fft.fft2(psi) * h)
        far = torch.fft.fft2(psi)
        amp = far.abs()
        if I is None:
            pats[b:b + len(ps)] = amp.square()
            continue
        root = I[b:b + len(ps)].double().sqrt()
        loss = loss + (root - amp).square().sum()
        chi = torch.fft.ifft2(far * torch.where(amp > thr, 1.0 - root / torch.where(amp > thr, amp, 1.0), 1.0)) * w ** 2
        at = ((ps[:, 0, None].long() + r)[:, :, None] * nx + (ps[:, 1, None].long() + r)[:, None, :]).reshape(-1)
        illum.index_add_(0, at, into[lowest].abs().square().reshape(-1))
        for l in range(L - 1, lowest - 1, -1):
            dX[l].index_add_(0, at, (into[l].conj() * chi).reshape(-1))
            chi = _windows(X[l], ps, w).conj() * chi
            if l > 0:
                chi = torch.fft.ifft2(torch.fft.fft2(chi) * h.conj())
        if lowest == 0:
            dprobe += chi.sum(0)
    return pats, loss, dX.reshape(L, *X[0].shape), dprobe, illum


def _phase(V):
    return torch.polar(torch.ones_like(V), SIGMA * V)


def _layer(case, probe, V, pos, I, l):
    X = _phase(V)
    _, loss, dX, _, illum = _pass(case, probe, X, pos, I, lowest=l)
    mu = 1.0 / (2 * SIGMA ** 2 * case["win"] ** 2 * illum.max())
    V = V.clone()
    V[l] -= mu * 2 * SIGMA * (X[l].conj() * dX[l]).imag
    return loss, mu, V


def _exact_scan(case, seed):
    kind, t = case["kind"], _inputs(case, seed)
    probe, pos, I = t["probe"].to(torch.complex128), t["pos"], t["I"]
    if case["param"] == "transmission":
        _, loss, dX, dp, _ = _pass(case, probe, t["V"].to(torch.complex128), pos, I)
        return {"loss": loss.reshape(1), "dV": dX, "dprobe": dp}
    V = t["V"].double()
    if kind == "forward":
        return {"I": _pass(case, probe, _phase(V), pos, None)[0]}
    if kind == "layer":
        loss, mu, V = _layer(case, probe, V, pos, I, case["layer"])
        return {"loss": loss.reshape(1), "mu": mu.reshape(1), "V": V}
    if kind == "reconstruct":
        history = []
        for _ in range(case["sweeps"]):
            for l in range(case["n_slices"]):
                loss, _, V = _layer(case, probe, V, pos, I, l)
                history.append(loss)
            for _ in range(case["probe_steps"]):
                _, loss, _, dp, _ = _pass(case, probe, _phase(V), pos, I)
                probe = probe - dp / (len(pos) * case["win"] ** 2)
                history.append(loss)
        history.append(_pass(case, probe, _phase(V), pos, I)[1])
        return {"history": torch.stack(history), "V": V, "probe": probe}
    X = _phase(V)
    _, loss, dX, dp, _ = _pass(case, probe, X, pos, I)
    dV = 2 * SIGMA * (X.conj() * dX).imag
    if kind == "autograd":   # torch's gradient of a complex argument is twice the Wirtinger derivative
        return {"loss": loss, "dV": dV, "dprobe": 2 * dp}
    return {"loss": loss.reshape(1), "dV": dV, "dprobe": dp}


def _exact_smd(case, seed):
    t = _smd_inputs(case, seed)
    n, M = case["n"], case["n_slices"]
    h = _fresnel(n, 2 * 5.6533 / 40, SMD_LAMBDA_A, 20.0, t["A"].device)
    probe, A, o = (t[k].to(torch.complex128) for k in ("probe", "A", "o"))
    lam, I = t["lam"][0], t["I"].double()
    P = torch.stack([torch.roll(probe, (int(a), int(b)), (0, 1)).reshape(-1) for a, b in t["shifts"].tolist()])
    U = torch.fft.fft2((P @ A).reshape(-1, n, n))   # A holds columns as rows
    amp, root, thr = U.abs(), I.sqrt(), ZERO_TAU * I.mean().sqrt()
    objective = 0.5 * (root - amp).square().sum()
    R = U * torch.where(amp > thr, 1.0 - root / torch.where(amp > thr, amp, 1.0), 1.0)
    mu = 1.0 / (n ** 2 * torch.fft.fft2(probe).abs().max() ** 2)
    A = A - mu * (P.conj().T @ (torch.fft.ifft2(R) * n ** 2).reshape(-1, n * n))

    def go(x, hh):
        return torch.fft.ifft2(torch.fft.fft2(x) * hh)

    new = []
    D = (lam * _transfer(o, h) - A).reshape(-1, n, n)
    before = 0.5 * D.abs().square().sum()
    e, into = torch.eye(n * n, dtype=o.dtype, device=o.device).reshape(-1, n, n), []
    for m in range(M):
        into.append(e)
        e = go(e * o[m], h)
    grads, back = [None] * M, D
    for m in range(M - 1, -1, -1):
        grads[m] = lam * (back * into[m].conj()).sum(0)
        back = go(back * o[m].conj(), h.conj())
    del e, into, back, D
    top = o.abs().reshape(M, -1).max(dim=1).values
    for m in range(M):
        c = lam * torch.prod(torch.cat([top[:m], top[m + 1:]]))
        x = o[m] - grads[m] / c ** 2
        new.append(x / x.abs().square().sum().sqrt())
    o = torch.stack(new)
    At = _transfer(o, h)
    lam = (A.conj() * At).sum().real / At.abs().square().sum()
    return {"objective": objective.reshape(1), "mu": mu.reshape(1), "before": before.reshape(1), "A": lam * At, "o": o,
            "lam": lam.reshape(1)}


def _bf16(x):
    return x.float().bfloat16().double()


def _exact_train(case, seed):
    """In 64 bits between the BF16 values that the network stores: its input, weights, activations and
    pre-activation gradients."""
    t = _net_inputs(case, seed)
    lay, n = _net_layout(case["n_slices"])
    p, L = t["p"].double(), case["n_slices"]
    weights = []
    a, acts, pres = _bf16(torch.cat([t["V"], t["G"]]))[None], [], []
    for i, (ci, co, x, y) in enumerate(lay):
        w = _bf16(p[x:y]).reshape(co, 3, 3, ci).permute(0, 3, 1, 2).contiguous()
        weights.append(w)
        acts.append(a)
        z = torch.nn.functional.conv2d(a, w, p[y:y + co], padding=1)
        pres.append(z)
        a = _bf16(torch.nn.functional.gelu(z))
    d = pres[-1] - t["target"].double()[None] / 0.5
    loss = d.square().mean()
    g, grad = _bf16(2.0 / d.numel() * d), torch.empty(n, dtype=torch.float64, device=p.device)
    for i in range(5, -1, -1):
        ci, co, x, y = lay[i]
        dw = torch.nn.grad.conv2d_weight(acts[i], weights[i].shape, g, padding=1)
        grad[x:y] = dw.permute(0, 2, 3, 1).reshape(-1)
        grad[y:y + co] = g.sum((0, 2, 3))
        if i:
            z = pres[i - 1]
            slope = 0.5 * (1 + torch.erf(z / math.sqrt(2.0))) + z * torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)
            g = _bf16(torch.nn.grad.conv2d_input(acts[i].shape, weights[i], g, padding=1) * slope)
    m = 0.9 * t["m"].double() + 0.1 * grad
    v = 0.999 * t["v"].double() + 0.001 * grad * grad
    p = p - 1e-4 * (m / (1 - 0.9 ** 100)) / ((v / (1 - 0.999 ** 100)).sqrt() + 1e-8)
    return {"loss": loss, "p": p, "m": m, "v": v}


def exact(case, seed):
    with torch.no_grad():
        return {"smd": _exact_smd, "train": _exact_train}.get(case["kind"], _exact_scan)(case, seed)
