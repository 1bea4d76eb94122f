"""D3Q27 steps on changing streams: the near pass, the particle kernel and the auxiliary kernel run on streams of the
context's own, beside the caller's, and the auxiliary kernel of a call's last step must be done before the next call's
particle kernel reads its inverse, whichever stream that call is on.  Calls of one and of several steps, the particle's
forces changed in between, against the same calls on the context's own stream, bit for bit."""
import numpy as np
import pytest

from lb_inputs import box, particle, random_quaternion, rng

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
L = pytest.importorskip("paper_2403_05443_gb300.lbsph")


@pytest.mark.parametrize("didt_mode", [0, 2])
def test_calls_on_changing_streams(didt_mode):
    g = rng(8)
    boxes = [box(32, 32, 32, 0.8, counter_force=1), box(24, 32, 28, 0.9, counter_force=1)]
    parts = [[particle((4.0, 2.5, 2.5), (0.3, 15.9, 31.8), random_quaternion(g), U=(0.03, 0, -0.02), density=3.0)],
             [particle((4.5, 3.0, 2.5), (12.1, 0.2, 13.7), random_quaternion(g), Om=(0.01, 0.02, 0))]]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    ft = g.normal(size=(12, 2, 6)) * 1e-3
    counts = [1, 1, 2, 1, 5, 1, 1, 3, 1, 1, 7, 1]

    def run(pick):
        sim = L.Simulation(boxes, parts, max_semi=5, lattice=27, didt_mode=didt_mode)
        for k, n in enumerate(counts):
            s = pick(k)
            sim.step(n, s)
            if s is not None:
                streams[k % 2].synchronize()
            sim.set_external(-1, ft[k], s)
            if s is not None:
                streams[k % 2].synchronize()
        return [sim.field(f, b) for f in ("df", "u", "solid") for b in (0, 1)] + [sim.records(b) for b in (0, 1)]

    for a, b in zip(run(lambda k: streams[k % 2].cuda_stream), run(lambda k: None)):
        assert np.array_equal(a, b) and np.isfinite(a.astype(float)).all() and a.any()
