"""The network's kernels start while the kernel before them may still be writing (programmatic launch).  What that one
writes must not be read by non-coherent loads (__ldg: read-only for the whole life of the reading kernel).  It may be a
caller's buffer as well: the prediction of one forward pass as the targets of the next call, all of it queued without
a wait, gives the same bits as with a wait after every call.

Every wait in them is bounded.  One that gives up must do so for the whole warp (lanes that part would meet at
different barriers), and the block must wait again for the copies and products it has in flight before it leaves; no
such wait can be made to run out here without holding up the GPU, so this is checked in the source."""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("kernel", ["net_kernel", "grad_kernel", "head_row"])
def test_no_non_coherent_load_in_kernels_that_start_early(kernel):
    with open(os.path.join(ROOT, "paper_2403_05443_gb300", "csrc", "mlp_kernel.cu")) as f:
        text = f.read()
    m = re.search(r"\n[^\n/]*\b%s\(.*?\n}\n" % kernel, text, re.S)
    assert m and "__ldg(" not in m.group(0)


def test_a_wait_that_gives_up_leaves_nothing_in_flight():
    with open(os.path.join(ROOT, "paper_2403_05443_gb300", "csrc", "mlp_kernel.cu")) as f:
        text = f.read()
    body = re.search(r"\n[^\n/]*\bgrad_kernel\(.*?\n}\n", text, re.S).group(0)
    bias, tiles = body.split("// ---- operands and place of this tile")
    # waits by a whole warp: decided together
    assert len(re.findall(r"__all_sync\(0xffffffffu, mbar_wait\(full", bias)) == 1
    assert len(re.findall(r"__all_sync\(0xffffffffu, use == 0 \|\| mbar_wait\(empty", tiles)) == 1
    # the second waits: the biases' copies; the last copies into every stage and the last product of a tile's
    assert re.search(r"if \(!ok\) \{[^}]*\(void\)mbar_wait\(full, 0u\);", bias)
    fail = tiles.split("if (fail) {", 1)[1].split("if (nrank > 1)", 1)[0]
    assert "k = max(0, issued - GST); k < issued; ++k) (void)mbar_wait(full + k % GST, (unsigned)(k / GST) & 1u)" in fail
    assert "(void)mbar_wait(empty + (issued - 1) % GST, (unsigned)((issued - 1) / GST) & 1u)" in fail


@pytest.mark.gpu
@pytest.mark.parametrize("n", [100, 1024, 1200])
def test_outputs_of_one_call_as_inputs_of_the_next(n):
    torch = pytest.importorskip("torch")
    SU = pytest.importorskip("paper_2403_05443_gb300.surrogate")
    g = np.random.default_rng(n)
    P = (0.05 * g.standard_normal(SU.LB_MLP_NPARAM)).astype(np.float32)
    x = torch.from_numpy(g.standard_normal((n, 8)).astype(np.float32)).cuda()

    def run(wait):
        net = SU.Surrogate(max_batch=n, params=P)
        R = torch.zeros((n, 36), device="cuda")
        loss, grad = torch.zeros(12, device="cuda"), torch.zeros((6, SU.LB_MLP_NPARAM), device="cuda")
        torch.cuda.synchronize()
        for k in range(6):
            SU.lb_mlp_forward(net.h, x.data_ptr(), n, None, R.data_ptr())
            if wait:
                torch.cuda.synchronize()
            # targets: the prediction itself; a step (Adam moves even where the gradient is tiny), and the loss after it
            SU.lb_mlp_train_step(net.h, x.data_ptr(), R.data_ptr(), n, 1e-2, loss.data_ptr() + 8 * k)
            if wait:
                torch.cuda.synchronize()
            SU.lb_mlp_loss_grad(net.h, x.data_ptr(), R.data_ptr(), n, loss.data_ptr() + 8 * k + 4, grad.data_ptr() + 4 * k * SU.LB_MLP_NPARAM)
            if wait:
                torch.cuda.synchronize()
        SU.lb_gemm_status()
        return R.cpu().numpy(), loss.cpu().numpy(), grad.cpu().numpy(), net.params()

    for a, b in zip(run(False), run(True)):
        assert np.array_equal(a, b) and np.isfinite(a).all()
