"""pty_profile_*: the stages of a pass cover all of its kernels."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,Nz,grads", [(64, 6, ("amp", "phase", "probe", "pos")), (64, 10, ("phase",)), (256, 4, ("phase", "probe"))])
def test_sparsity_term_is_in_a_stage(N, Nz, grads):
    """Objects of 6 and 10 Mi voxels (the object's gradient beside the probe's in one launch, and by itself), one position:
    the sparsity term's passes over the object are a third of the call or more, so the stages' sum is close to the
    call's time only with them in it."""
    from paper_2505_07814_gb300 import _lib
    from paper_2505_07814_gb300.ptycho import Geometry, Params, Ptycho
    H = 1024
    geom = Geometry(N=N, M=1, Nz=Nz, H=H, W=H, Ntot=1, dx=0.1, lam=0.025, grads=grads, w_sparse=0.1, p_sparse=1.5)
    f = dict(dtype=torch.float32, device="cuda")
    params = Params(torch.ones((Nz, H, H), **f), torch.full((Nz, H, H), 0.1, **f), torch.ones((1, N, N), dtype=torch.complex64, device="cuda"),
                    torch.full((1, 2), 30.25, **f), torch.zeros((1, 2), **f), torch.ones(1, **f))
    pt, I, out = Ptycho(geom, 1), torch.ones((1, N, N), **f), params.zeros_like()
    pt.loss_grad(params, [0], I, grads=out)
    begin, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    calls = 20
    idx = torch.zeros(1, dtype=torch.int32, device="cuda")
    _lib.pty_profile_enable(True)
    try:
        torch.cuda.synchronize()
        torch.cuda._sleep(20_000_000)  # the launches queue up behind it: no gaps between the calls' kernels
        begin.record()
        for _ in range(calls):
            pt.loss_grad(params, idx, I, grads=out)
        end.record()
        torch.cuda.synchronize()
        n, ms = _lib.pty_profile_read()
    finally:
        _lib.pty_profile_enable(False)
    assert n == calls and pt.status() == 0
    total = begin.elapsed_time(end)
    assert sum(ms.values()) >= 0.85 * total, (sum(ms.values()), total, ms)
