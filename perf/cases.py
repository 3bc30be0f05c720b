"""The work that users of this framework have it do, as cases that can be timed.

A case is one pass through the public Python entry points: the forward model, loss and gradients of a
batch of scan positions (`Ptycho.loss_grad`), an optimiser iteration (`step`), the differentiable
forward model under torch autograd (`forward_model`), pattern simulation (`Ptycho.forward`), the
constraints after an iteration (`constrain`), and training and inference of the learned initialiser
(`Cnn`).  Sizes are those of the repository's workloads (`synth.workload`), its tests and its benchmark.

Inputs are a reconstruction in progress: measured patterns simulated from a true object, probe and scan
(Poisson counts, or the expected patterns of a noise-free simulation), and an estimate of all of them
as it is in an early iteration.  `exact` evaluates the same model in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2505_07814_gb300.cnn import LAYER_CHANNELS, Cnn, he_init
from paper_2505_07814_gb300.ptycho import Adam, Geometry, Params, Ptycho, constrain, forward_model, step

DX = float(np.float32(0.1))  # angstrom per pixel, as the library receives it
LAM = float(np.float32(0.025079340450548))  # 200 kV, angstrom
OBJECT_PROBE_POS = ("amp", "phase", "probe", "pos")
# what a run refines: the usual four, those and the tilt, or the slice spacing too (one number that is a
# sum of millions of terms of both signs: listed once, where they do not cancel)
REFINED = {"usual": OBJECT_PROBE_POS, "tilt": OBJECT_PROBE_POS + ("tilt",), "all": OBJECT_PROBE_POS + ("tilt", "dz")}
ALL = REFINED["all"]
# the estimate: an early iteration, off by half of the phase, 20 angstrom of defocus, a fifth of the
# probe's amplitude, 0.2 angstrom of position, 3 mrad of tilt and half of the slice spacing
ESTIMATE = dict(phase=0.5, amp_noise=0.05, phase_noise=0.01, defocus=70.0, probe_noise=0.2, pos=2.0, tilt=3e-3, dz=3.0)
TRUTH = dict(absorption=0.1, defocus=50.0, dz=2.0)
COUNTS = 0.6  # electrons per detector pixel
EPS = float(np.float32(1e-6))  # stabiliser inside the Poisson logarithm
S_IN = 0.2  # the initialiser's input scale
LR = {"amp": 5e-4, "phase": 5e-4, "probe": 1e-4, "pos": 5e-4}
LARGEST = 256 * 12 * 20 * 256 * 256  # positions x modes x slices x window pixels of the largest listed case


def _wave(name, call, N, M, Nz, H, W, scan, B, **more):
    c = {"name": name, "kind": "wave", "call": call, "N": N, "M": M, "Nz": Nz, "H": H, "W": W, "scan": scan, "B": B,
         "loss": "gaussian", "data": "counts", "grads": "tilt", "sparse": 0.0, "stride": 1, "fft": "fp32"}
    c.update(more)
    return c


def _constrain(name, N, M, Nz, H, W):
    return {"name": name, "kind": "constrain", "N": N, "M": M, "Nz": Nz, "H": H, "W": W}


def _cnn(name, call, S, B):
    return {"name": name, "kind": "cnn", "call": call, "S": S, "B": B}


def listed():
    return [
        # the smallest calls: 2D ptychography (64 x 64 window, one mode, one slice) in batches of 16,
        # where launches and latency count
        _wave("single_slice_b16", "loss_grad", 64, 1, 1, 128, 128, 16, 16),
        # the same reconstruction with its whole 16 x 16 scan as one batch
        _wave("single_slice_b256", "loss_grad", 64, 1, 1, 128, 128, 16, 256),
        # the iteration of a published reconstruction's shape: 12 modes, 6 slices of 614 x 614, batches
        # of 16, object, probe and positions refined by Adam, sparsity term on
        _wave("iteration_12mode_b16", "step", 128, 12, 6, 614, 614, 128, 16, grads="usual", sparse=0.1),
        # ordinary multislice work: 6 modes, 8 slices of 512 x 512, all six gradients, batches of 512, Poisson
        # likelihood
        _wave("multislice_b512", "loss_grad", 128, 6, 8, 512, 512, 64, 512, grads="all", loss="poisson",
              data="expected"),
        # simulation of patterns (training pairs of the initialiser, simulated data sets)
        _wave("simulate_b512", "forward", 128, 6, 8, 512, 512, 64, 512),
        # the split-precision transforms on the tensor cores at the accuracy of FP32
        _wave("multislice_bf16x3_b64", "loss_grad", 128, 6, 8, 512, 512, 64, 64, fft="bf16x3"),
        # the largest: 256 x 256 windows, 12 modes, 20 slices of 1024 x 1024, batches of 256
        _wave("large_window_b256", "loss_grad", 256, 12, 20, 1024, 1024, 64, 256),
        # large windows under a memory budget (segments of 5 slices re-run in the adjoint), a loss of
        # the user's own through torch autograd
        _wave("large_window_autograd_b16", "autograd", 256, 12, 20, 1024, 1024, 64, 16, stride=5),
        # the constraints after an iteration, every one of them: a large volume with power-of-two
        # sides, and the ragged sides that a scan's extent usually gives
        _constrain("constrain_20x1024x1024", 256, 12, 20, 1024, 1024),
        _constrain("constrain_6x614x614", 128, 12, 6, 614, 614),
        # the learned initialiser: a training step and inference on 256 patterns of 128 x 128
        _cnn("initialiser_train_b256", "train", 128, 256),
        _cnn("initialiser_predict_b256", "predict", 128, 256),
    ]


def _spread(rng, lo, hi):
    """An integer in [lo, hi], spread over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["wave"] * 8 + ["constrain"] * 2 + ["cnn"] * 2)
    if kind == "cnn":
        S = rng.choice([64, 96, 128])
        c = _cnn("", rng.choice(["train", "predict"]), S, _spread(rng, 16, 256))
    elif kind == "constrain":
        N = rng.choice([64, 128, 256])
        H, W = (rng.choice([512, 1024]) if rng.random() < 0.3 else _spread(rng, N, 1024) for _ in range(2))
        c = _constrain("", N, rng.randint(2, 12), rng.randint(2, 20), H, W)
    else:
        call = rng.choice(["loss_grad", "loss_grad", "loss_grad", "step", "forward", "autograd"])
        N = rng.choice([64, 128, 128, 256])
        M, Nz = _spread(rng, 1, 12), _spread(rng, 1, 20)
        B = _spread(rng, 8, 256 if N == 256 else 512)
        fft = "fp32"
        if call == "loss_grad" and N < 256 and rng.random() < 0.15:
            fft, B = "bf16x3", min(B, 64)
        scan = rng.choice([32, 48, 64])
        H, W = (min(1024, N + 10 + 2 * scan + rng.randint(0, 300)) for _ in range(2))
        while B * M * Nz * N * N > LARGEST:
            B = B // 2
        # (one or two modes leave interference zeros, where the Poisson weight d / I has no stable value)
        loss = rng.choice(["gaussian", "poisson"]) if M > 2 else "gaussian"
        c = _wave("", call, N, M, Nz, H, W, scan, B, loss=loss, data="counts" if loss == "gaussian" else "expected",
                  grads=rng.choice(["usual", "tilt"]), fft=fft)
        if call == "step":
            c.update(grads="usual", sparse=rng.choice([0.0, 0.1]))
        if fft == "fp32" and call in ("loss_grad", "autograd") and Nz >= 4 and rng.random() < 0.25:
            c["stride"] = rng.randint(2, Nz - 1)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, shape):
    return torch.rand(shape, generator=g, device="cuda")


def _randn(g, shape):
    return torch.randn(shape, generator=g, device="cuda")


def _atoms(g, Nz, H, W):
    """Phase of Nz slices of Gaussian atoms (0.4 angstrom wide, 0.3 rad high, 0.1 per square angstrom)."""
    hit = (_rand(g, (Nz, H, W)) < 0.1 * DX * DX).float()
    fy, fx = torch.fft.fftfreq(H, device="cuda")[:, None], torch.fft.rfftfreq(W, device="cuda")[None]
    sigma = 0.4 / DX
    blur = 0.3 * 2 * math.pi * sigma ** 2 * torch.exp(-2 * (math.pi * sigma) ** 2 * (fy ** 2 + fx ** 2))
    return torch.fft.irfft2(torch.fft.rfft2(hit) * blur, s=(H, W)).clamp_min(0.0)


def _probe(g, N, M, defocus=TRUTH["defocus"]):
    """Orthogonal probe modes: a 20 mrad aperture, defocused, times low-order monomials; the
    first mode holds 0.6 of the dose, the others a geometric share of the rest."""
    k = torch.fft.fftfreq(N, d=DX, device="cuda", dtype=torch.float64)
    kk = k[:, None] ** 2 + k[None] ** 2
    base = torch.fft.fftshift(torch.fft.ifft2((kk.sqrt() <= 20e-3 / LAM) * torch.exp(-1j * math.pi * LAM * defocus * kk)))
    r = (torch.arange(N, device="cuda", dtype=torch.float64) - N / 2) * DX
    monos = [(a, n - a) for n in range(5) for a in range(n, -1, -1)][:M]
    modes = []
    for a, b in monos:
        c = 1.0 + 0.05 * torch.view_as_complex(_randn(g, (2,)).double())
        v = base * r[:, None] ** a * r[None] ** b * c
        for u in modes:
            v = v - (u.conj() * v).sum() * u
        modes.append(v / v.abs().square().sum().sqrt())
    power = [1.0] if M == 1 else [0.6] + [0.4 * 0.5 ** i / (2 - 0.5 ** (M - 2)) for i in range(M - 1)]
    return torch.stack([m * math.sqrt(p * COUNTS * N * N) for m, p in zip(modes, power)]).to(torch.complex64)


def _patterns(patches, probe, frac, tilt, dz):
    """The multislice model: patches [b, Nz, N, N] complex, probe [M, N, N], frac / tilt [b, 2], dz [1];
    DC-centred intensities [b, N, N] in the precision of the inputs."""
    N, Nz, rd = probe.shape[-1], patches.shape[1], frac.dtype
    f = torch.fft.fftfreq(N, device=probe.device, dtype=rd)
    ramp = frac[:, 0, None, None] * f[:, None] + frac[:, 1, None, None] * f[None]
    wave = torch.fft.ifft2(torch.fft.fft2(probe)[None] * torch.exp(-2j * math.pi * ramp)[:, None])
    k = f / DX
    t = torch.tan(tilt)
    arg = -LAM * dz * (k[:, None] ** 2 + k[None] ** 2) + 2 * dz * (t[:, 0, None, None] * k[:, None] + t[:, 1, None, None] * k[None])
    prop = torch.exp(1j * math.pi * arg)[:, None]
    for s in range(Nz):
        wave = wave * patches[:, None, s]
        if s + 1 < Nz:
            wave = torch.fft.ifft2(torch.fft.fft2(wave) * prop)
    far = torch.fft.fft2(wave, norm="ortho")
    return torch.fft.fftshift((far.real ** 2 + far.imag ** 2).sum(1), dim=(-2, -1))


def _chunk(c, per_value):
    """Positions per chunk of the plain torch model that keep it under some 12 GB."""
    return max(1, min(c["B"], int(12e9 / (per_value * c["M"] * (c["Nz"] + 2) * c["N"] ** 2))))


def _cut(T, corners, N):
    return torch.stack([T[:, r:r + N, q:q + N] for r, q in corners])


def _inputs(c, seed):
    """Everything that a program has in hand: the estimate, the batch, the measured patterns."""
    g = _gen(seed)
    N, M, Nz, H, W, B, n = c["N"], c["M"], c["Nz"], c["H"], c["W"], c["B"], c["scan"]
    phase_t = _atoms(g, Nz, H, W)
    state = g.get_state()
    probe_t = _probe(g, N, M)
    g.set_state(state)
    probe_e = _probe(g, N, M, ESTIMATE["defocus"])  # the same modes, wrongly focused
    ax = [torch.linspace(4.0, L - N - 4.0, n, device="cuda") for L in (H, W)]
    pos_t = torch.stack(torch.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 2) + 0.6 * (_rand(g, (n * n, 2)) - 0.5)
    tilt_t = torch.tensor([0.5e-3, -0.3e-3], device="cuda").expand(n * n, 2)
    dz_t = torch.tensor([TRUTH["dz"]], device="cuda")
    idx = torch.randperm(n * n, generator=g, device="cuda")[:B].to(torch.int32)
    e = ESTIMATE
    est = Params(amp=1.0 + e["amp_noise"] * _randn(g, (Nz, H, W)),
                 phase=e["phase"] * phase_t + e["phase_noise"] * _randn(g, (Nz, H, W)),
                 probe=probe_e * (1.0 + e["probe_noise"] * torch.view_as_complex(_randn(g, (M, N, N, 2)))),
                 pos=pos_t + e["pos"] * (2 * _rand(g, pos_t.shape) - 1), tilt=tilt_t + e["tilt"] * _randn(g, pos_t.shape),
                 dz=torch.tensor([e["dz"]], device="cuda"))
    meas = None
    if c["call"] != "forward":
        T, rows = torch.polar(1.0 - TRUTH["absorption"] / 0.3 * phase_t, phase_t), []
        sel, per = idx.long(), _chunk(c, 40)
        for s in range(0, B, per):
            p = pos_t[sel[s:s + per]]
            at = torch.round(p)
            rows.append(_patterns(_cut(T, at.long().tolist(), N), probe_t, p - at, tilt_t[sel[s:s + per]], dz_t))
        rows = torch.cat(rows)
        if c["data"] == "counts":
            rows = torch.poisson(rows, generator=g)
        meas = rows[torch.arange(n * n, device="cuda") % B]  # the scan's other patterns: like these
        meas[sel] = rows
    return est, idx, meas


def _grads_of(c):
    return REFINED[c["grads"]]


def _own_loss(I, rows):
    """A loss of the user's own for the autograd case: amplitude residuals, softened at zero."""
    return ((I + 0.1).sqrt() - (rows + 0.1).sqrt()).square().mean()


def _plain(c, est, idx, meas, dtype):
    """Loss and gradients of the batch by torch autograd in `dtype` (float32 or float64)."""
    cd = torch.complex128 if dtype == torch.float64 else torch.complex64
    N, B, Nz = c["N"], c["B"], c["Nz"]
    sel = idx.long()
    amp, phase = est.amp.to(dtype), est.phase.to(dtype)
    unit = torch.polar(torch.ones_like(phase), phase)
    T = amp * unit
    probe = est.probe.to(cd).requires_grad_(True)
    pos, tilt = est.pos.to(dtype), est.tilt.to(dtype)
    dz = est.dz.to(dtype).requires_grad_(True)
    corners = torch.round(est.pos[sel]).long().tolist()
    per = _chunk(c, 120 if dtype == torch.float32 else 240)

    def model(s, grad):
        p = pos[sel[s:s + per]]
        leaves = [_cut(T, corners[s:s + per], N), p - torch.round(p), tilt[sel[s:s + per]]]
        leaves = [x.detach().requires_grad_(grad) for x in leaves]
        return leaves, _patterns(leaves[0], probe, leaves[1], leaves[2], dz)

    if c["call"] == "forward":
        with torch.no_grad():
            return torch.cat([model(s, False)[1] for s in range(0, B, per)])
    rows = meas[sel].to(dtype)
    S = rows.sum() if c["loss"] == "poisson" else rows.sqrt().sum()
    Q = 0.0
    if c["loss"] == "gaussian" and c["call"] != "autograd":
        with torch.no_grad():
            for s in range(0, B, per):
                Q = Q + (model(s, False)[1].sqrt() - rows[s:s + per].sqrt()).square().sum()
    out = Params(torch.zeros_like(T), None, torch.zeros_like(probe), torch.zeros_like(pos), torch.zeros_like(tilt),
                 torch.zeros_like(dz))
    loss = torch.zeros((), dtype=dtype, device="cuda")
    for s in range(0, B, per):
        leaves, I = model(s, True)
        d = rows[s:s + per]
        if c["call"] == "autograd":
            part = _own_loss(I, d) * (d.shape[0] / B)
            loss += part.detach()
        elif c["loss"] == "poisson":
            part = -(d * torch.log(I + EPS) - I).sum() / S
            loss += part.detach()
        else:
            part = (I.sqrt() - d.sqrt()).square().sum() * (math.sqrt(d[0].numel() * B) / (2 * Q.sqrt() * S))
        gp, gf, gt, gprobe, gdz = torch.autograd.grad(part, leaves + [probe, dz], allow_unused=True, materialize_grads=True)
        for i, (r, q) in enumerate(corners[s:s + per]):
            out.amp[:, r:r + N, q:q + N] += gp[i]
        out.pos[sel[s:s + per]] = gf
        out.tilt[sel[s:s + per]] = gt
        out.probe += gprobe
        out.dz += gdz
    if c["loss"] == "gaussian" and c["call"] != "autograd":
        loss = (Q * N * N * B).sqrt() / S
    gT = out.amp
    out.amp = (unit.conj() * gT).real
    out.phase = (T.conj() * gT).imag
    if c["sparse"]:
        cover = torch.zeros(T.shape[1:], dtype=dtype, device="cuda")
        for r, q in corners:
            cover[r:r + N, q:q + N] += 1
        n = B * Nz * N * N
        loss = loss + c["sparse"] * (cover * phase.abs()).sum() / n
        out.phase = out.phase + c["sparse"] * cover * phase.sign() / n
    out.probe, out.dz = out.probe.detach(), out.dz.detach()
    return loss.detach().reshape(1), out


def _moments(c, est, idx, meas):
    """Adam's moments of a run in progress: near the present gradient and its square."""
    _, g = _plain(c, est, idx, meas, torch.float32)
    m, v = {}, {}
    for name in ALL:
        x = getattr(g, name)
        x = torch.view_as_real(x) if x.is_complex() else x
        m[name] = 0.5 * x
        v[name] = x.square() + x.square().mean() + 1e-20
    return m, v


def _conv_inputs(c, seed):
    g = _gen(seed)
    S, B = c["S"], c["B"]
    r = torch.arange(S, device="cuda") - S / 2
    rr = (r[:, None] ** 2 + r[None] ** 2).sqrt()
    disc = 1.0 / (1.0 + torch.exp((rr - 0.08 * S) / (0.02 * S))) + 0.02 * torch.exp(-((rr / (0.2 * S)) ** 2))
    speckle = torch.nn.functional.avg_pool2d(_rand(g, (B, 1, S, S)), 5, 1, 2)[:, 0] * 2
    I = torch.poisson(300.0 * disc * speckle, generator=g)
    Y = torch.nn.functional.avg_pool2d(_randn(g, (B, 2, S // 2, S // 2)), 9, 1, 4).permute(0, 2, 3, 1).contiguous()
    params = torch.tensor(he_init(2000 + seed % 1000), device="cuda")
    params = params + 0.01 * _randn(g, params.shape)
    m, v = 1e-3 * _randn(g, params.shape), 1e-4 * (0.5 + _rand(g, params.shape))
    return I, Y, params, m, v


def _constrain_inputs(c, seed):
    g = _gen(seed)
    M, N = c["M"], c["N"]
    phase = _atoms(g, c["Nz"], c["H"], c["W"]) + 0.01 * _randn(g, (c["Nz"], c["H"], c["W"]))
    amp = 1.0 + 0.02 * _randn(g, phase.shape)
    mix = torch.eye(M, device="cuda") + 0.05 * torch.view_as_complex(_randn(g, (M, M, 2)))
    probe = torch.einsum("mk,kij->mij", mix, _probe(g, N, M)).contiguous()
    return amp, phase, probe


# one set of settings: regularised along the beam, blurred by one slice, phase >= 0, modes orthogonal
CONSTRAIN = dict(phase_positivity=1.0, rz_sigma=1.0, rz_relax=1.0, kz_beta=1.0, kz_alpha=0.01, kz_relax=1.0,
                 orthogonalize_probe=True)


# ---------------------------------------------------------------------------------------------
# The cases' interface
# ---------------------------------------------------------------------------------------------
def prepare(case, seed):
    c = case
    if c["kind"] == "cnn":
        I, Y, params, m, v = _conv_inputs(c, seed)
        net = Cnn(S=c["S"], max_batch=c["B"], s_in=S_IN, params=params)
        net.m.copy_(m)
        net.v.copy_(v)
        net.step_count = 100
        return {"case": c, "net": net, "I": I, "Y": Y, "loss": torch.zeros(1, device="cuda")}
    if c["kind"] == "constrain":
        amp, phase, probe = _constrain_inputs(c, seed)
        geom = Geometry(N=c["N"], M=c["M"], Nz=c["Nz"], H=c["H"], W=c["W"], Ntot=1, dx=DX, lam=LAM, grads=())
        pos, tilt, dz = (torch.zeros(n, device="cuda") for n in ((1, 2), (1, 2), 1))
        params = Params(amp, phase, probe.clone(), pos, tilt, dz + 2.0)
        return {"case": c, "pt": Ptycho(geom, 1), "params": params, "probe": probe}
    est, idx, meas = _inputs(c, seed)
    geom = Geometry(N=c["N"], M=c["M"], Nz=c["Nz"], H=c["H"], W=c["W"], Ntot=c["scan"] ** 2, dx=DX, lam=LAM,
                    loss=c["loss"], grads=() if c["call"] == "forward" else _grads_of(c), ckpt_stride=c["stride"],
                    fft=c["fft"], w_sparse=c["sparse"])
    s = {"case": c, "pt": Ptycho(geom, c["B"]), "params": est, "idx": idx, "meas": meas,
         "loss": torch.zeros(1, device="cuda")}
    if c["call"] in ("loss_grad", "step"):
        s["grads"] = est.zeros_like()
    if c["call"] == "step":
        m, v = _moments(c, est, idx, meas)
        s["adam"] = Adam(est, LR)
        for name in ALL:
            for dst, src in ((s["adam"].m, m), (s["adam"].v, v)):
                dst = getattr(dst, name)
                (torch.view_as_real(dst) if dst.is_complex() else dst).copy_(src[name])
        s["adam"].t = 100
    if c["call"] == "forward":
        s["out"] = torch.empty((c["B"], c["N"], c["N"]), device="cuda")
    if c["call"] == "autograd":
        s["rows"] = meas[idx.long()]
        s["leaves"] = [getattr(est, n).requires_grad_(True) for n in _grads_of(c)]
        del s["meas"]
    return s


def run(state):
    c = state["case"]
    if c["kind"] == "cnn":
        net = state["net"]
        if c["call"] == "predict":
            return net.predict(state["I"])
        # the loss goes into the run's float32 history
        state["loss"].copy_(net.train_step(state["I"], state["Y"], lr=1e-3))
        return {"loss": state["loss"], "grad": net.grad, "params": net.params}
    p = state["params"]
    if c["kind"] == "constrain":
        p.probe.copy_(state["probe"])  # as an optimiser's update leaves it: not orthogonal
        constrain(state["pt"], p, **CONSTRAIN)
        return {"amp": p.amp, "phase": p.phase, "probe": p.probe}
    pt, idx = state["pt"], state["idx"]
    if c["call"] == "forward":
        return pt.forward(p, idx, out=state["out"])
    if c["call"] == "autograd":
        loss = _own_loss(forward_model(pt, p, idx), state["rows"])
        return [loss.detach().reshape(1), *torch.autograd.grad(loss, state["leaves"])]
    if c["call"] == "step":
        state["loss"].copy_(step(pt, p, state["grads"], state["adam"], idx, state["meas"]))
        return {"loss": state["loss"], **{n: getattr(state["grads"], n) for n in OBJECT_PROBE_POS},
                **{"new_" + n: getattr(p, n) for n in OBJECT_PROBE_POS}}
    loss, g = pt.loss_grad(p, idx, state["meas"], grads=state["grads"])
    state["loss"].copy_(loss)
    return {"loss": state["loss"], **{n: getattr(g, n) for n in _grads_of(c)}}


def work(case):
    c = case
    if c["kind"] == "cnn":
        S, B = c["S"], c["B"]
        sides = (S // 2, S // 4, S // 8, S // 16, S // 8, S // 2)
        macs = [9 * ic * oc * h * h for (ic, oc), h in zip(LAYER_CHANNELS[:5], sides)]
        # the last layer, behind a fourfold upsampling, needs its channel products once per coarse pixel
        macs.append(9 * 2 * 256 * (S // 8) ** 2)
        n = sum(9 * ic * oc + oc for ic, oc in LAYER_CHANNELS)
        io = 4 * B * (S * S + 2 * (S // 2) ** 2)
        if c["call"] == "predict":
            return {"bytes": io + 4 * n, "flops": 2.0 * B * sum(macs)}
        return {"bytes": io + 4 * n * 7, "flops": 2.0 * B * (3 * sum(macs) - macs[0])}
    N, M, Nz, H, W = c["N"], c["M"], c["Nz"], c["H"], c["W"]
    obj, probe = 4 * Nz * H * W, 8 * M * N * N
    if c["kind"] == "constrain":
        # two 3D transforms of the object as one complex volume, and the modes' Gram matrix and mixing
        flops = 2 * 5.0 * Nz * H * W * math.log2(Nz * H * W) + 2 * 8.0 * M * M * N * N
        return {"bytes": 2 * 2 * obj + 2 * probe, "flops": flops}
    B, NN = c["B"], N * N
    fft = 5.0 * NN * math.log2(NN)
    fwd = 2 * Nz * fft + NN * (12 + 6 * Nz + 12 * (Nz - 1) + 5)
    if c["call"] == "forward":
        return {"bytes": 2 * obj + probe + 4 * B * NN, "flops": B * M * fwd}
    adj = 2 * Nz * fft + NN * (4 + 12 * Nz + 16 * (Nz - 1) + 22)
    nbytes = 2 * 2 * obj + 2 * probe + 4 * B * NN
    if c["call"] == "step":  # the moments read and written, the parameters written
        nbytes += 5 * (2 * obj + probe)
    return {"bytes": nbytes, "flops": B * M * (fwd + adj)}


def _exact_cnn(c, seed):
    I, Y, params, m, v = _conv_inputs(c, seed)
    # rounded as the network's storage is not: plain 64-bit convolutions of the given parameters
    flat = params.double().requires_grad_(True)
    x = (float(np.float32(S_IN)) * torch.log1p(I.double()))[:, None]
    o = 0
    for l, (ic, oc) in enumerate(LAYER_CHANNELS):
        w = flat[o:o + 9 * ic * oc].reshape(oc, 3, 3, ic).permute(0, 3, 1, 2)
        b = flat[o + 9 * ic * oc:o + 9 * ic * oc + oc]
        o += 9 * ic * oc + oc
        if l >= 4:
            x = torch.nn.functional.interpolate(x, scale_factor=2 if l == 4 else 4, mode="nearest")
        x = torch.nn.functional.conv2d(x, w, b, stride=2 if l < 4 else 1, padding=1)
        x = torch.relu(x) if l < 5 else x
    pred = x.permute(0, 2, 3, 1)
    if c["call"] == "predict":
        return pred.detach().contiguous()
    loss = (pred - Y.double()).square().mean()
    g, = torch.autograd.grad(loss, flat)
    new = _adam(flat.detach(), g, m.double(), v.double(), 101, 1e-3)
    return {"loss": loss.detach().reshape(1), "grad": g, "params": new}


def _adam(x, g, m, v, t, lr, b1=0.9, b2=0.999, eps=1e-8):
    if x.is_complex():
        return torch.view_as_complex(_adam(torch.view_as_real(x), torch.view_as_real(g), m, v, t, lr).contiguous())
    m = b1 * m + (1 - b1) * g
    v = b2 * v + (1 - b2) * g * g
    return x - lr * (m / (1 - b1 ** t)) / ((v / (1 - b2 ** t)).sqrt() + eps)


def _exact_constrain(c, seed):
    amp, phase, probe = (x.to(torch.complex128 if x.is_complex() else torch.float64) for x in _constrain_inputs(c, seed))
    M, Nz, H, W = c["M"], c["Nz"], c["H"], c["W"]
    A = probe.reshape(M, -1)
    lam, U = torch.linalg.eigh(A @ A.conj().T)
    U = U[:, lam.argsort(descending=True)]
    big = U.gather(0, U.abs().argmax(0, keepdim=True))
    new_probe = ((U * (big.conj() / big.abs())).conj().T @ A).reshape(probe.shape)
    freq = lambda n, d: torch.fft.fftfreq(n, d=d, device="cuda", dtype=torch.float64)  # noqa: E731
    kr2 = freq(H, DX)[:, None] ** 2 + freq(W, DX)[None] ** 2
    kz2 = freq(Nz, 2.0)[:, None, None] ** 2
    alpha = float(np.float32(CONSTRAIN["kz_alpha"]))
    Wa = (1 - (2 / math.pi) * torch.atan(CONSTRAIN["kz_beta"] ** 2 * kz2 / (kr2 + 1e-3))) * torch.exp(-alpha * kr2)
    s = torch.arange(Nz, device="cuda")
    d = (s[:, None] - s[None]).abs()
    taps = torch.where(d <= math.ceil(4 * CONSTRAIN["rz_sigma"]), torch.exp(-0.5 * (d / CONSTRAIN["rz_sigma"]).double() ** 2), 0.0)
    taps = taps / taps.sum(1, keepdim=True)
    out = [torch.einsum("st,tij->sij", taps, torch.fft.ifftn(torch.fft.fftn(x) * Wa).real) for x in (amp, phase)]
    return {"amp": out[0], "phase": out[1].clamp_min(0.0), "probe": new_probe}


def exact(case, seed):
    c = case
    if c["kind"] == "cnn":
        return _exact_cnn(c, seed)
    if c["kind"] == "constrain":
        return _exact_constrain(c, seed)
    est, idx, meas = _inputs(c, seed)
    got = _plain(c, est, idx, meas, torch.float64)
    if c["call"] == "forward":
        return got
    loss, g = got
    if c["call"] == "autograd":
        return [loss, *(getattr(g, n) for n in _grads_of(c))]
    if c["call"] == "loss_grad":
        return {"loss": loss, **{n: getattr(g, n) for n in _grads_of(c)}}
    m, v = _moments(c, est, idx, meas)
    new = {}
    for n in OBJECT_PROBE_POS:
        x = getattr(est, n)
        x = x.to(torch.complex128 if x.is_complex() else torch.float64)
        new["new_" + n] = _adam(x, getattr(g, n), m[n].double(), v[n].double(), 101, LR[n])
    return {"loss": loss, **{n: getattr(g, n) for n in OBJECT_PROBE_POS}, **new}
