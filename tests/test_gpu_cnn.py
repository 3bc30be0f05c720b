"""Learned-initialiser kernels (include/pty_cnn.h) against the FP64 CNN oracle with the same bf16
storage points.

Layer by layer: each layer's oracle is fed the GPU's own stored inputs (activations, gradients), so
its FP64 result and the GPU's FP32 result differ only by FP32 rounding.  Where they are rounded to
bf16 they then agree exactly except where the value lies within that rounding of a bf16 tie: those
elements may differ by one bf16 unit and must be rare (<= 0.2%).  FP32 outputs (predictions, weight
and bias gradients) agree to relative L2 <= 2e-5.

End to end, the few one-unit flips of early layers spread through every later layer, so the whole
network is held to the bf16 level instead: relative L2 <= 4e-3 (about 2 units of bf16 rounding,
2^-9 each) on predictions and <= 1e-2 on gradients.

The last test trains the network on forward-model pairs and compares the reconstruction started
from its stitched prediction with the one from the paper's flat start.
"""
import numpy as np
import pytest

from oracle import cnn as C
from oracle import ptycho as O
from tests.cases import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_PRED = 4e-3
TOL_GRAD = 1e-2
TOL_F32 = 2e-5
FLIP_FRAC = 2e-3


def _net(S, B, seed=3):
    from paper_2505_07814_gb300.cnn import Cnn, he_init
    p = he_init(seed)
    p[C.param_count() - 2:] = [0.05, -0.02]  # nonzero output biases
    return Cnn(S=S, max_batch=B, params=torch.tensor(p, device="cuda")), p.astype(np.float64)


def _data(S, B, seed=0):
    rng = np.random.default_rng(seed)
    I = rng.gamma(1.5, 40.0, (B, S, S)).astype(np.float32)
    I[:, :S // 4, :] *= 0.01  # dim region: small log values next to bright ones
    Y = (0.2 * rng.standard_normal((B, S // 2, S // 2, 2))).astype(np.float32)
    return I, Y


def _layer_slices():
    out, o = [], 0
    for ic, oc, _, _, _ in C.LAYERS:
        out.append((slice(o, o + 9 * ic * oc), slice(o + 9 * ic * oc, o + 9 * ic * oc + oc)))
        o += 9 * ic * oc + oc
    return out


@pytest.mark.parametrize("S,B", [(128, 3), (64, 5), (32, 2)])
def test_forward_matches_oracle(S, B):
    net, p = _net(S, B)
    I, _ = _data(S, B)
    pred = net.predict(torch.tensor(I, device="cuda"))
    torch.cuda.synchronize()
    ref, _ = C.forward(p, I, net.s_in, bf=True)
    assert rel_l2(pred.cpu().numpy(), ref) <= TOL_PRED


@pytest.mark.parametrize("S,B", [(128, 2), (64, 3)])
def test_loss_and_gradients_match_oracle(S, B):
    net, p = _net(S, B, seed=4)
    I, Y = _data(S, B, seed=1)
    It, Yt = torch.tensor(I, device="cuda"), torch.tensor(Y, device="cuda")
    pred = torch.empty((B, S // 2, S // 2, 2), device="cuda")
    loss, grad = net.loss_grad(It, Yt, pred=pred)
    torch.cuda.synchronize()
    ref_loss, ref_grad = C.loss_and_grad(p, I, Y, net.s_in, bf=True)
    assert abs(loss.item() - ref_loss) <= 1e-3 * ref_loss
    g = grad.cpu().numpy()
    for k, (ws, bs) in enumerate(_layer_slices()):
        assert rel_l2(g[ws], ref_grad[ws]) <= TOL_GRAD, ("weights", k + 1, rel_l2(g[ws], ref_grad[ws]))
        assert rel_l2(g[bs], ref_grad[bs]) <= TOL_GRAD, ("bias", k + 1, rel_l2(g[bs], ref_grad[bs]))
    # the same call twice gives the same loss (fixed-order FP64 reduction)
    loss2, _ = net.loss_grad(It, Yt)
    assert loss2.item() == loss.item()


def test_empty_batch_and_bad_arguments():
    from paper_2505_07814_gb300 import _lib
    net, _ = _net(64, 2)
    I = torch.empty((0, 64, 64), device="cuda")
    Y = torch.empty((0, 32, 32, 2), device="cuda")
    loss, grad = net.loss_grad(I, Y)
    torch.cuda.synchronize()
    assert loss.item() == 0.0 and float(grad.abs().max()) == 0.0
    with pytest.raises(_lib.PtyError):
        _lib.pty_cnn_workspace_size(40, 2)
    with pytest.raises(_lib.PtyError):  # workspace too small
        _lib.pty_cnn_forward(64, 2, net.params.data_ptr(), I.data_ptr(), 0.2, Y.data_ptr(), net.ws.data_ptr(), 1024,
                             None)


def test_adam_matches_torch():
    from paper_2505_07814_gb300.cnn import Cnn
    net, _ = _net(32, 1)
    p0 = net.params.clone()
    ref = torch.nn.Parameter(p0.clone())
    opt = torch.optim.Adam([ref], lr=3e-3, betas=(0.9, 0.999), eps=1e-8)
    g = torch.randn_like(p0)
    from paper_2505_07814_gb300 import _lib
    s = torch.cuda.current_stream().cuda_stream
    for step in range(1, 4):
        gs = g * step
        _lib.pty_cnn_adam(net.params.data_ptr(), net.m.data_ptr(), net.v.data_ptr(), gs.data_ptr(), step, 3e-3, 0.9,
                          0.999, 1e-8, s)
        ref.grad = gs.clone()
        opt.step()
    torch.cuda.synchronize()
    assert float((net.params - ref.detach()).abs().max()) <= 1e-6 * float(p0.abs().max()) + 1e-7


def test_targets_and_stitching_match_oracle():
    from paper_2505_07814_gb300 import cnn
    rng = np.random.default_rng(11)
    S, Nz, H, W = 32, 3, 90, 100
    amp = np.exp(-rng.uniform(0, 0.1, (Nz, H, W))).astype(np.float32)
    phase = rng.uniform(0, 0.3, (Nz, H, W)).astype(np.float32)
    pos = np.array([[0.0, 0.0], [10.4, 20.6], [30.5, 41.5], [58.0, 68.0], [31.5, 12.49]], dtype=np.float32)
    idx = np.array([4, 0, 2, 1, 3], dtype=np.int32)
    dev = "cuda"
    t = lambda x: torch.tensor(x, device=dev)
    Y = cnn.targets(S, t(amp), t(phase), t(pos), t(idx)).cpu().numpy()
    corners = [tuple(O.crop_index(pos[j])[0]) for j in idx]
    ref = C.targets(amp, phase, corners, S)
    np.testing.assert_allclose(Y, ref, rtol=1e-5, atol=1e-5)
    wgt = rng.uniform(0.2, 1.0, (S // 2, S // 2)).astype(np.float32)
    pred = (0.1 * rng.standard_normal((5, S // 2, S // 2, 2))).astype(np.float32)
    st = cnn.Stitcher(S, Nz, H, W, t(wgt), device=dev)
    st.add(t(pred), t(pos), t(idx))
    a, ph = st.finish()
    ra, rph = C.stitch(pred.astype(np.float64), corners, wgt.astype(np.float64), H, W, S, Nz)
    np.testing.assert_allclose(ph.cpu().numpy(), rph, rtol=1e-5, atol=1e-6)
    np.testing.assert_allclose(a.cpu().numpy(), ra, rtol=1e-5, atol=1e-6)


def test_training_reduces_the_loss():
    """A fixed batch of patterns with targets that depend on them is fitted by 60 Adam steps."""
    S, B = 64, 16
    net, _ = _net(S, B, seed=5)
    I, _ = _data(S, B, seed=2)
    # targets: a smooth function of the pattern's mean intensity (learnable from the input)
    m = np.log1p(I).mean(axis=(1, 2))
    Y = np.zeros((B, S // 2, S // 2, 2), dtype=np.float32)
    Y[..., 0] = (m - m.mean())[:, None, None]
    It, Yt = torch.tensor(I, device="cuda"), torch.tensor(Y, device="cuda")
    l0 = net.loss_grad(It, Yt)[0].item()
    for _ in range(60):
        net.train_step(It, Yt, lr=1e-3)
    l1 = net.loss_grad(It, Yt)[0].item()
    assert l1 < 0.3 * l0, (l0, l1)


def _np(t):
    return t.detach().cpu().numpy().astype(np.float64)


def _assert_bf16_close(got, ref, what):
    """Equal except for rare one-unit bf16 differences (or differences far below the scale)."""
    d = np.abs(got - ref)
    scale = np.abs(ref).max()
    ulp = np.maximum(np.abs(got), np.abs(ref)) * 2.0 ** -7
    bad = d > np.maximum(ulp * 1.0001, 1e-6 * scale)
    assert not bad.any(), (what, int(bad.sum()), float(d.max()))
    frac = float((d > 1e-6 * scale).mean())
    assert frac <= FLIP_FRAC, (what, frac)


@pytest.mark.parametrize("S,B", [(128, 2), (64, 3)])
def test_each_layer_matches_oracle_on_the_gpu_inputs(S, B):
    net, p = _net(S, B, seed=6)
    I, Y = _data(S, B, seed=3)
    It, Yt = torch.tensor(I, device="cuda"), torch.tensor(Y, device="cuda")
    pred = torch.empty((B, S // 2, S // 2, 2), device="cuda")
    net.loss_grad(It, Yt, pred=pred)
    torch.cuda.synchronize()
    grad = _np(net.grad)
    pred = _np(pred)
    wb = C.unpack(p)
    acts = [C.net_input(I, net.s_in)] + [_np(net.state(B, l, "act")) for l in range(1, 6)]
    dz = {l: _np(net.state(B, l, "dz")) for l in range(1, 7)}
    # forward, one layer at a time from the GPU's stored inputs
    for l in range(1, 6):
        _, _, stride, up, _ = C.LAYERS[l - 1]
        ref = C.bf16(np.maximum(C.conv_forward(acts[l - 1], C.bf16(wb[l - 1][0]), wb[l - 1][1], stride, up), 0.0))
        _assert_bf16_close(acts[l], ref, ("act", l))
    ref = C.conv_forward(acts[5], C.bf16(wb[5][0]), wb[5][1], 1, 4)
    assert rel_l2(pred, ref) <= TOL_F32
    # loss gradient at the output
    _assert_bf16_close(dz[6], C.bf16(2.0 * (pred - Y) / pred.size), "dz6")
    # backward, one layer at a time from the GPU's stored gradients
    for l, (ws, bs) in reversed(list(enumerate(_layer_slices(), start=1))):
        _, _, stride, up, _ = C.LAYERS[l - 1]
        dx, dw, db = C.conv_backward(acts[l - 1], C.bf16(wb[l - 1][0]), stride, up, dz[l])
        assert rel_l2(grad[ws], dw.ravel()) <= TOL_F32, ("dW", l, rel_l2(grad[ws], dw.ravel()))
        assert rel_l2(grad[bs], db) <= TOL_F32, ("db", l, rel_l2(grad[bs], db))
        if l > 1:
            _assert_bf16_close(dz[l - 1], C.bf16(dx * (acts[l - 1] > 0)), ("dz", l - 1))


@pytest.mark.parametrize("S,B", [(48, 7), (80, 3), (112, 2)])
def test_each_layer_at_tile_edges(S, B):
    """Row counts that end inside the GEMMs' 128-row tiles, in every parity class of the input gradients."""
    test_each_layer_matches_oracle_on_the_gpu_inputs(S, B)


def test_smallest_network_matches_oracle():
    test_forward_matches_oracle(16, 1)


def test_wait_that_runs_out_returns_etimeout_and_the_next_call_is_clean():
    from paper_2505_07814_gb300 import _lib
    net, _ = _net(64, 3)
    I, Y = (torch.tensor(x, device="cuda") for x in _data(64, 3))
    want, pred = torch.empty((3, 32, 32, 2), device="cuda"), torch.empty((3, 32, 32, 2), device="cuda")

    def status():
        return _lib.pty_status(net.ws.data_ptr(), torch.cuda.current_stream().cuda_stream)

    net.loss_grad(I, Y, pred=want)
    assert status() == 0
    try:
        _lib.pty_set_wait_limit(0)
        net.loss_grad(I, Y, pred=pred)
        st = status()
    finally:
        _lib.pty_set_wait_limit(-1)
    assert st >= 0 and st & _lib.PTY_ETIMEOUT, st
    net.loss_grad(I, Y, pred=pred)
    assert status() == 0 and torch.equal(pred, want)


def test_learned_start_reaches_target_nmse_sooner_than_flat_start():
    """Trained on 16384 forward-model pairs from four random volumes (not the test object), the
    network's stitched start is closer to the truth than the flat start and the reconstruction
    from it reaches object NMSE <= 0.05 in fewer Adam batches (same lr, batch, seed)."""
    from paper_2505_07814_gb300 import learned_init as L
    from paper_2505_07814_gb300.cnn import Cnn
    prob = L.problem("c2")
    amp_f, ph_f = L.flat_object(prob)
    I, Y = L.training_set(prob, n_objects=4, per_object=4096)
    net = Cnn(S=128, max_batch=256)
    L.train(net, I, Y, epochs=4, batch=256, lr=1e-3)
    del I, Y
    amp_c, ph_c = L.initial_object(net, prob)
    # the package's NMSE is the oracle's definition
    r0, r1, c0, c1 = prob.roi
    e_pkg = L.nmse(ph_c, prob.truth.phase, prob.roi)
    e_orc = C.nmse(_np(ph_c).sum(0), _np(prob.truth.phase).sum(0), prob.roi)
    assert abs(e_pkg - e_orc) <= 1e-9 * max(e_orc, 1.0)
    assert L.nmse(ph_f, prob.truth.phase, prob.roi) > 0.99
    assert e_pkg < 0.8
    lr = {"phase": 1e-3}
    h_flat, _ = L.reconstruct(prob, amp_f, ph_f, iters=4, batch=64, lr=lr)
    h_cnn, _ = L.reconstruct(prob, amp_c, ph_c, iters=4, batch=64, lr=lr)
    assert h_flat[-1][1] <= 0.05 and h_cnn[-1][1] <= 0.05
    assert h_cnn[-1][0] < h_flat[-1][0], (h_cnn[-1], h_flat[-1])
