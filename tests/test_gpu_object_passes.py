"""The object's passes (transmission, dL/dT, dL/damp and dL/dphase): four elements at a time where the arrays allow it, one
otherwise, in a launch with the probe's transforms up to some object size and by themselves above it."""
import dataclasses

import numpy as np
import pytest

from tests.cases import make_case
from tests.test_gpu_parity import _check_all, _gpu, _np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
GRADS = ("amp", "phase", "probe", "pos", "tilt", "dz")


def _offset(t, shift=1):
    """The same values in a view that starts `shift` elements into its buffer."""
    buf = torch.zeros(t.numel() + shift, dtype=t.dtype, device=t.device)
    view = buf[shift:].view(t.shape)
    view.copy_(t)
    return view


def _close(a, b, bar):
    a, b = _np(a).ravel(), _np(b).ravel()
    assert np.linalg.norm(a - b) <= bar * np.linalg.norm(b), np.linalg.norm(a - b) / np.linalg.norm(b)


# step 5, pads 7 / 10 give odd plane sizes; (8, 8) and step 8 sides that are multiples of eight
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("N,kw", [(64, dict(step=8, pad=(8, 8))), (64, dict(step=5, pad=(7, 10))), (128, dict(step=8, pad=(8, 8))),
                                  (256, dict(step=8, pad=(8, 8)))])
def test_arrays_off_a_16_byte_boundary(N, kw, accumulate):
    """Only which arrays are read four at a time changes: patterns and loss are equal, gradients to the last bits of
    their atomic sums (1e-6)."""
    case = make_case(N=N, M=2, Nz=2, scan=(2, 2), seed=61, **kw)
    idx = [0, 1, 2, 3]
    pt, params, I_meas = _gpu(case)
    out = params.zeros_like()
    for n in GRADS:
        getattr(out, n).fill_(0.25 if accumulate else float("nan"))
    off_p, off_g = params.zeros_like(), params.zeros_like()
    for n in GRADS:
        setattr(off_p, n, _offset(getattr(params, n)))
        setattr(off_g, n, _offset(getattr(out, n)))
    loss, _ = pt.loss_grad(params, idx, I_meas, grads=out, accumulate=accumulate)
    loss, I = loss.item(), pt.forward(params, idx)
    loss2, _ = pt.loss_grad(off_p, idx, _offset(I_meas), grads=off_g, accumulate=accumulate)
    assert pt.status() == 0 and loss2.item() == loss
    assert torch.equal(pt.forward(off_p, idx), I)
    for n in GRADS:
        _close(getattr(off_g, n), getattr(out, n), 1e-6)


# 8 Mi = 2^23 voxels: just below and just above, plane sizes that are multiples of four (2896^2, 2898^2) and that are not
@pytest.mark.parametrize("H,W", [(2896, 2896), (2895, 2895), (2898, 2898), (2898, 2895)])
@pytest.mark.parametrize("N,Nz", [(64, 1), (128, 1)])
def test_object_sizes_around_the_shared_launch(N, Nz, H, W):
    """A small case, and the same case in the corner of a large object of ones: the gradients are the small one's there and
    zero elsewhere."""
    from paper_2505_07814_gb300.ptycho import Params, Ptycho
    case = make_case(N=N, M=2, Nz=Nz, scan=(2, 2), seed=62)
    idx = [0, 1, 2, 3]
    pt, params, I_meas, _ = _check_all(case, idx)
    h, w = case.geom.H, case.geom.W
    _, small = pt.loss_grad(params, idx, I_meas)
    small_loss = pt.loss.item()
    big = Ptycho(dataclasses.replace(pt.geom, H=H, W=W), len(idx))
    amp, phase = torch.ones((Nz, H, W), device="cuda"), torch.zeros((Nz, H, W), device="cuda")
    amp[:, :h, :w], phase[:, :h, :w] = params.amp, params.phase
    p = Params(amp, phase, params.probe, params.pos, params.tilt, params.dz)
    out = p.zeros_like()
    out.amp.fill_(float("nan"))
    out.phase.fill_(float("nan"))
    loss, _ = big.loss_grad(p, idx, I_meas, grads=out)
    assert big.status() == 0 and loss.item() == small_loss
    for n in ("amp", "phase"):
        g = getattr(out, n)
        _close(g[:, :h, :w], getattr(small, n), 1e-6)
        g[:, :h, :w] = 0
        assert not g.any()
    for n in ("probe", "pos", "tilt", "dz"):
        a, b = getattr(out, n), getattr(small, n)
        if n in ("tilt", "dz") and Nz == 1:
            assert not a.any()
        else:
            _close(a, b, 1e-6)
