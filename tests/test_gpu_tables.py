"""The per-wave tables (shift ramps, propagator factors, dz and tilt factors) at arguments far from the usual
ones: propagator phases of hundreds of turns, tilts of tens of milliradians, sub-pixel shifts at the edge.

The tables carry their phase as a pair of floats, so its error stays at 48 bits of the argument and the
usual FP32 bars hold (1e-5 on patterns and loss, 1e-4 on gradients); a phase rounded to one float would be
off by 1e-5 turns at these arguments.  The loss is the Gaussian one: the Poisson weights d / I of a single
mode's interference zeros make the gradients miss 1e-4 in any FP32 evaluation, whatever the tables.
"""
import dataclasses

import numpy as np
import pytest

from oracle import ptycho as O
from tests.cases import f32, make_case, oracle_grads, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,dz,global_tilt", [(64, 400.0, False), (128, 250.0, False), (64, 37.5, True), (256, 150.0, False)])
def test_tables_at_large_arguments(N, dz, global_tilt):
    from paper_2505_07814_gb300.ptycho import Geometry, Params, Ptycho
    case = make_case(N=N, M=1, Nz=2, scan=(1, 3), seed=31, dz=dz, global_tilt=global_tilt, loss=O.GAUSSIAN)
    rng = np.random.default_rng(5)
    case.tilt = f32(case.tilt + 0.04 * rng.uniform(-1, 1, np.shape(case.tilt)))
    case.pos = f32(np.round(case.pos) + 0.498 * np.where(rng.random(case.pos.shape) < 0.5, -1, 1))
    g = case.geom
    geom = Geometry(N=g.N, M=g.M, Nz=g.Nz, H=g.H, W=g.W, Ntot=case.Ntot, dx=g.dx, lam=g.lam, eps=g.eps, loss="gaussian",
                    global_tilt=g.global_tilt)
    t = dict(dtype=torch.float32, device="cuda")
    params = Params(amp=torch.tensor(case.amp, **t), phase=torch.tensor(case.phase, **t),
                    probe=torch.tensor(case.probe, dtype=torch.complex64, device="cuda"), pos=torch.tensor(case.pos, **t),
                    tilt=torch.tensor(case.tilt, **t), dz=torch.tensor([case.dz], **t))
    idx = list(range(case.Ntot))
    pt = Ptycho(geom, case.Ntot)
    I = torch.empty((len(idx), N, N), **t)
    loss, grads = pt.loss_grad(params, idx, torch.tensor(case.I_meas, **t), I_model=I)
    torch.cuda.synchronize()
    assert pt.status() == 0
    ref = oracle_grads(case, idx)
    assert rel_l2(I.cpu().numpy(), ref.I_model) <= 1e-5
    assert abs(loss.item() - ref.loss) <= 1e-5 * abs(ref.loss)
    for name in ("amp", "phase", "probe", "pos", "tilt"):
        assert rel_l2(getattr(grads, name).cpu().numpy(), getattr(ref, name)) <= 1e-4, name


# Far beyond a sampled propagation: phases of up to pi lam dz k^2 / pi = 0.63 dz per axis, 9400 to 250000 half turns,
# so that the low float of a table's phase is up to 1 / 64 of a half turn.  A white probe puts the waves at every
# frequency.  48 bits of 250000 are 1e-9, below the FP32 bars.
FAR = [(64, 1.5e4, True), (128, 1.2e5, False), (256, 4e5, False), (64, -4e5, False)]


def far_case(N, dz, global_tilt):
    case = make_case(N=N, M=1, Nz=2, scan=(1, 2), seed=41, global_tilt=global_tilt, loss=O.GAUSSIAN)
    rng = np.random.default_rng(6)
    white = rng.standard_normal(case.probe.shape) + 1j * rng.standard_normal(case.probe.shape)
    case.probe = np.asarray(white * (np.linalg.norm(case.probe) / np.linalg.norm(white)), np.complex64).astype(np.complex128)
    case.tilt = f32(0.02 * rng.uniform(-1, 1, np.shape(case.tilt)))
    case.dz = float(np.float32(dz))
    # the pixel size as the library receives it: 0.1 itself is off by 1.5e-8, 1e-3 half turns of the smallest case's phase
    case.geom = dataclasses.replace(case.geom, dx=float(np.float32(case.geom.dx)))
    return case


@pytest.mark.parametrize("N,dz,global_tilt", FAR)
def test_tables_far_beyond_sampled_propagations(N, dz, global_tilt):
    from paper_2505_07814_gb300.ptycho import Geometry, Params, Ptycho
    case = far_case(N, dz, global_tilt)
    g = case.geom
    geom = Geometry(N=g.N, M=g.M, Nz=g.Nz, H=g.H, W=g.W, Ntot=case.Ntot, dx=g.dx, lam=g.lam, eps=g.eps, loss="gaussian",
                    global_tilt=g.global_tilt)
    t = dict(dtype=torch.float32, device="cuda")
    params = Params(amp=torch.tensor(case.amp, **t), phase=torch.tensor(case.phase, **t),
                    probe=torch.tensor(case.probe, dtype=torch.complex64, device="cuda"), pos=torch.tensor(case.pos, **t),
                    tilt=torch.tensor(case.tilt, **t), dz=torch.tensor([case.dz], **t))
    idx = list(range(case.Ntot))
    pt = Ptycho(geom, case.Ntot)
    I = torch.empty((len(idx), N, N), **t)
    loss, grads = pt.loss_grad(params, idx, torch.tensor(case.I_meas, **t), I_model=I)
    torch.cuda.synchronize()
    assert pt.status() == 0
    ref = oracle_grads(case, idx)
    assert rel_l2(I.cpu().numpy(), ref.I_model) <= 1e-5
    assert abs(loss.item() - ref.loss) <= 1e-5 * abs(ref.loss)
    for name in ("amp", "phase", "probe", "pos", "tilt"):
        assert rel_l2(getattr(grads, name).cpu().numpy(), getattr(ref, name)) <= 1e-4, name
    assert abs(grads.dz.item() - ref.dz) <= 1e-4 * abs(ref.dz)
