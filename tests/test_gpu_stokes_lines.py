"""lb_stokes_field on edges that take every kind of line transform (radices 8, 4, 2, 3, 5,
primes by their definition, lines long enough that fewer of them share a block), with
outputs that start on any byte and without the density, against oracle/warmstart.py.

Bar: three FP32 passes each way; a radix-r butterfly by its definition adds at most r
rounding errors of 6e-8 (r <= 101 here: 6e-6), the others a few: 1e-5 normwise."""
import numpy as np
import pytest

from lb_inputs import box, particle, random_quaternion, rng
from oracle import warmstart as W
from parity_util import normwise

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
L = pytest.importorskip("paper_2403_05443_gb300.lbsph")


@pytest.mark.parametrize("shape,tau,shift,density", [
    ((20, 22, 26), 0.8, 0, True),           # 4 x 5, 2 x 11, 2 x 13
    ((28, 35, 50), 1.2, 4, True),           # 4 x 7, 5 x 7, 2 x 5 x 5
    ((44, 101, 25), 0.7, 0, False),         # 4 x 11, a prime, 5 x 5
    ((24, 20, 320), 0.9, 0, True),          # 8 x 3, 4 x 5, 8 x 8 x 5
    ((48, 16, 27), 1.0, 2, True),           # 16 x 3, 4 x 4, 3 x 3 x 3; not aligned to the element
])
def test_stokes_field_for_every_line_length(shape, tau, shift, density):
    nx, ny, nz = shape
    g = rng(5)
    b = box(nx, ny, nz, tau, counter_force=1)
    p = [particle((3.0, 2.0, 2.0), (0.4 * nx, 0.3 * ny, 0.6 * nz), random_quaternion(g), F_ext=(2e-4, -1e-4, 5e-5))]
    sim = L.Simulation([b], [p], max_semi=3)
    N = nx * ny * nz
    raw = torch.zeros(16 * N + 16, dtype=torch.uint8, device="cuda")
    at = raw.data_ptr() + shift
    L.lb_stokes_field(sim.ctx, 0, at, at + 12 * N if density else None)
    out = raw.cpu().numpy()[shift:shift + 16 * N].copy().view(np.float32)
    ref, dref = W.stokes_field(nx, ny, nz, sim.field("solid"), [q["F_ext"] for q in p], (tau - 0.5) / 3.0, counter=True,
                               density=True, tau=tau, rho0=1.0)
    assert normwise(out[:3 * N].reshape(3, nz, ny, nx), ref) <= 1e-5
    if density:
        assert normwise(out[3 * N:].reshape(nz, ny, nx), dref) <= 1e-5
    else:
        assert not out[3 * N:].any()
