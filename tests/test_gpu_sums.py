"""Batch sums beyond the range of a float: every summand fits a float, a CTA's sum does not.

The sums are kept as pairs of floats; one that leaves their range has to come out as its FP64 value."""
import dataclasses

import numpy as np
import pytest

from oracle import ptycho as O
from tests.cases import f32, make_case
from tests.test_gpu_parity import _gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [64, 128, 256])
def test_loss_of_patterns_whose_sums_exceed_a_float(N):
    """Poisson loss -Y / S with counts around 2e35: S and Y of 32 detector rows are above 3.4e38.  32 or more rows of N pixels
    summed in FP32 a few at a time keep the loss at the FP32 bar of 1e-5."""
    case = make_case(N=N, M=1, Nz=1, scan=(1, 2), seed=51)
    case.I_meas = f32(2e35 * np.random.default_rng(1).uniform(0.5, 1.5, case.I_meas.shape))
    pt, params, I_meas = _gpu(case)
    loss, _ = pt.loss_grad(params, [0, 1], I_meas)
    I = O.model_patterns(case.geom, case.amp, case.phase, case.probe, case.pos, case.tilt, case.dz, [0, 1])
    ref = O.loss_value(case.geom, np.asarray(I), case.I_meas)
    assert pt.status() == 0 and np.isfinite(ref)
    assert abs(loss.item() - ref) <= 1e-5 * abs(ref), (loss.item(), ref)


@pytest.mark.parametrize("N", [64, 128, 256])
def test_adjoint_partial_that_exceeds_a_float(N):
    """dL/d dz of one pattern is 1e39, made of threads' parts below 3.4e38, and the batch holds the pattern twice with dL/dI
    of either sign: the two waves do the same arithmetic with opposite signs, so the sum is exactly zero."""
    case = make_case(N=N, M=1, Nz=2, scan=(1, 1), seed=9)
    case.geom = dataclasses.replace(case.geom, lam=float(np.float32(1000 * case.geom.lam)))  # the same propagator at dz / 1000
    case.dz = float(np.float32(case.dz / 1000))
    case.tilt = np.zeros_like(case.tilt)
    h = 1e-4 * case.dz
    I = [O.model_patterns(case.geom, case.amp, case.phase, case.probe, case.pos, case.tilt, case.dz + s, [0])[0] for s in (h, -h)]
    d = (I[0] - I[1]) / (2 * h)  # the steepest dL/dI: dL/d dz = sum d^2
    d *= 1e39 / np.square(d).sum()
    assert np.abs(d).max() < 1e37
    pt, params, _ = _gpu(case, grads=("dz",), max_batch=2)
    pt.forward_save(params, [0, 0])
    g = pt.backward(params, [0, 0], torch.tensor(np.stack([d, -d]), dtype=torch.float32, device="cuda"))
    assert pt.status() == 0
    assert g.dz.item() == 0.0
    half = torch.tensor(np.stack([d, -0.9 * d]), dtype=torch.float32, device="cuda")  # 1e39 - 0.9e39: fits a float again
    pt.forward_save(params, [0, 0])
    assert abs(pt.backward(params, [0, 0], half).dz.item() - 1e38) <= 1e-3 * 1e38
