"""The digits of lb_stokes_field: the per-mode solve carries FP32 terms in two-FP32 sums, and what is left must be the
rounding of the FP32 transforms.  Near tau = 1/2 the longitudinal part of a mode cancels to nu k^2 of its terms, so
digits lost in the sums or in the two solves show there first (solved as one system in FP64 from FP32 terms, the error was
1.6e-6 at tau = 0.52, 3e-6 at 0.505 and 2e-5 at 0.501).

Bar, normwise against oracle/warmstart.py: an FFT of N points and back passes every value through 2 log2 N butterfly
levels; one rounding of 2^-24 at each, all in one direction: 2 log2(N) 2^-24 (2.1e-6 at 64^3)."""
import math

import pytest

from lb_inputs import box, particle, random_quaternion, rng
from oracle import warmstart as W
from parity_util import normwise

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
L = pytest.importorskip("paper_2403_05443_gb300.lbsph")


@pytest.mark.parametrize("shape", [(64, 64, 64), (48, 50, 54), (128, 32, 32), (32, 36, 250)])
@pytest.mark.parametrize("tau", [0.501, 0.505, 0.52, 0.8, 1.45])
def test_error_is_the_transforms_rounding(shape, tau):
    nx, ny, nz = shape
    N = nx * ny * nz
    b = box(nx, ny, nz, tau, counter_force=1)
    p = [particle((3.0, 2.0, 2.0), (0.4 * nx, 0.3 * ny, 0.6 * nz), random_quaternion(rng(5)), F_ext=(2e-4, -1e-4, 5e-5))]
    sim = L.Simulation([b], [p], max_semi=3)
    out = torch.zeros(4 * N, device="cuda")
    L.lb_stokes_field(sim.ctx, 0, out.data_ptr(), out.data_ptr() + 12 * N)
    ref, dref = W.stokes_field(nx, ny, nz, sim.field("solid"), [q["F_ext"] for q in p], (tau - 0.5) / 3.0, counter=True,
                               density=True, tau=tau, rho0=1.0)
    a, bar = out.cpu().numpy(), 2.0 * math.log2(N) * 2.0 ** -24
    assert normwise(a[:3 * N].reshape(ref.shape), ref) <= bar
    assert normwise(a[3 * N:].reshape(dref.shape), dref, floor=0.0) <= bar
