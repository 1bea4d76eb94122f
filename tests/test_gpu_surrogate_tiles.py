"""The network's kernels work on tiles of 128 samples, sum over up to 8 tiles in the
samples' order and over more tiles in four parts: loss, gradients and one Adam step
at the edges of those ranges, with inputs that do and do not start on a 16-byte
boundary, against oracle/surrogate.py with the BF16 rounding of the CUDA path.

Bars as in test_gpu_surrogate.py: gradients 5e-3 normwise per block (BF16
rounding-boundary flips), the loss 2e-4; an Adam step's first update is lr times the
gradient's sign where the gradient is not small, so within 2e-2 lr there.
"""
import numpy as np
import pytest

from oracle import surrogate as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
SU = pytest.importorskip("paper_2403_05443_gb300.surrogate")


def _offset(a, shift):
    """Device copy of a (FP32) that starts `shift` floats into its allocation."""
    t = torch.zeros(a.size + shift, dtype=torch.float32, device="cuda")
    t[shift:] = torch.from_numpy(np.ascontiguousarray(a, np.float32).reshape(-1)).cuda()
    return t, t.data_ptr() + 4 * shift


@pytest.mark.parametrize("n,shift", [(1, 0), (128, 1), (129, 0), (1024, 0), (1025, 3), (4096, 0)])
def test_loss_gradients_and_step_at_tile_edges(n, shift):
    g = np.random.default_rng(n)
    P = {"W1": g.normal(0, 0.35, (256, 16)), "b1": g.normal(0, 0.1, 256), "W2": g.normal(0, 0.06, (256, 256)),
         "b2": g.normal(0, 0.1, 256), "W3": g.normal(0, 0.06, (32, 256)), "b3": g.normal(0, 0.3, 32)}
    P["W1"][:, 8:], P["W3"][21:], P["b3"][21:] = 0.0, 0.0, 0.0
    p = S.pack(P).astype(np.float32)
    x = g.normal(0, 1, (n, 8)).astype(np.float32)
    A = g.normal(0, 1, (n, 6, 6))
    Rt = (np.einsum("nik,njk->nij", A, A) / 6 + np.eye(6)).astype(np.float32)
    lref, gref = S.loss_grad(p.astype(np.float64), x.astype(np.float64), Rt.astype(np.float64), emulate=True)
    net = SU.Surrogate(max_batch=n, params=p)
    (xt, xp), (rt, rp) = _offset(x, shift), _offset(Rt, shift)
    loss = torch.zeros(3, device="cuda")
    grad, gp = _offset(np.zeros(SU.LB_MLP_NPARAM, np.float32), shift)
    SU.lb_mlp_loss_grad(net.h, xp, rp, n, loss.data_ptr(), gp)
    SU.lb_mlp_loss_grad(net.h, xp, rp, n, loss.data_ptr() + 4)          # the loss alone
    SU.lb_mlp_train_step(net.h, xp, rp, n, 1e-3, loss.data_ptr() + 8)
    SU.lb_gemm_status()
    got, ref = SU.unpack(grad.cpu().numpy()[shift:].astype(np.float64)), SU.unpack(gref)
    for k in ref:
        assert np.abs(got[k] - ref[k]).max() <= 5e-3 * np.abs(ref[k]).max(), k
    assert np.all(np.abs(loss.cpu().numpy() - lref) <= 2e-4 * lref)
    step = S.adam_step(p.astype(np.float64), gref, 0.0, 0.0, 1, 1e-3)[0]
    big = np.abs(gref) > 0.05 * np.abs(gref).max()
    assert np.abs(net.params() - step)[big].max() <= 2e-2 * 1e-3
    assert np.abs(net.params() - step).max() <= 2.0 * 1e-3 + 1e-7
    assert xt is not None and rt is not None
