"""More particles in a box than a warp has lanes: the bulk pass and the field read-back look at the redo cubes of 32
particles at a time, one per lane, and a warp may meet several cubes (rows of 16 nodes: eight rows to a warp, cubes of
10 nodes every 16 along y) from different lanes, of the first 32 or of the rest.  36 small spheroids, the first ones
across the faces in y and z, moving fast enough to cover and uncover nodes.

FP32 against the oracle, bars as in test_gpu_parity.py (maps bit for bit, fields, forces and poses 1e-5).  16-bit storage against the FP32 run: a step rounds every population once, by at
most 2^-11 (FP16) or 2^-8 (BF16) of its size, and the collision mixes them with weights of sum below 4: 4 steps times
that, normwise.  A boundary node written by the bulk pass is off by the populations themselves."""
import numpy as np
import pytest

from lb_inputs import box, particle, random_quaternion, rng
from oracle import oracle as O
from parity_util import normwise, oracle_df_gpu_layout

pytestmark = pytest.mark.gpu

L = pytest.importorskip("paper_2403_05443_gb300.lbsph")

NX, NY, NZ = 16, 48, 168


def _case(n=36):
    g = rng(41)
    parts = []
    for k in range(n):
        c = np.array([8.0, 0.1 + 16 * (k % 3), 0.2 + 14 * (k // 3)]) + g.uniform(-0.3, 0.3, 3)
        v = g.normal(size=3)
        parts.append(particle((1.9, 1.4, 1.3), c % [NX, NY, NZ], random_quaternion(g), U=list(0.06 * v / np.linalg.norm(v)),
                              F_ext=list(g.normal(size=3) * 1e-4)))
    return box(NX, NY, NZ, 0.9, counter_force=1), parts


@pytest.mark.parametrize("steps", [1, 8])
def test_36_particles_match_the_oracle(steps):
    b, parts = _case()
    sim = L.Simulation([b], [parts], max_semi=2)
    orc = O.Sim(b, parts, nthreads=8)
    assert np.array_equal(sim.field("solid"), orc.owner())
    sim.step(steps)
    orc.step(steps)
    own = orc.owner()
    assert np.array_equal(sim.field("solid"), own) and len(np.unique(own)) == 37
    assert normwise(sim.field("df"), oracle_df_gpu_layout(orc)) <= 1e-5
    rho, u = orc.moments()
    rho = np.asarray(rho).reshape(own.shape) - b["rho0"]
    rho[own != 0] = 0.0
    assert normwise(sim.field("rho"), rho) <= 1e-5
    assert normwise(sim.field("u"), np.moveaxis(u, -1, 0)) <= 1e-5
    rec = sim.records()
    ref = [orc.particle(k) for k in range(36)]
    assert normwise(rec[:, 6:9], np.array([r["F"] for r in ref])) <= 1e-5
    assert normwise(rec[:, 9:12], np.array([r["T"] for r in ref])) <= 1e-5
    for k, r in enumerate(ref):
        assert np.abs(rec[k, 18:21] - r["x"]).max() <= 1e-5 * 0.06 * steps + 1e-9, k


@pytest.mark.parametrize("prec,eps", [(L.LB_FP16, 2.0 ** -11), (L.LB_BF16, 2.0 ** -8)])
def test_36_particles_in_16_bit_storage(prec, eps):
    steps = 8
    b, parts = _case()
    ref = L.Simulation([b], [parts], max_semi=2)
    sim = L.Simulation([b], [parts], max_semi=2, precision=prec)
    for s in (ref, sim):
        s.step(steps)
    assert np.array_equal(sim.field("solid"), ref.field("solid"))
    for name in ("df", "u"):
        assert normwise(sim.field(name), ref.field(name).astype(np.float64)) <= 4 * steps * eps, name


@pytest.mark.parametrize("n,ok", [(4, True), (5, False)])
def test_particles_that_one_read_back_tile_may_meet(n, ok):
    """A 256-quad tile meets at most four particles (LB_ECAPACITY): cubes side by side along x, in one tile's rows."""
    b = box(16 * n, 16, 16, 1.0)
    sim = L.Simulation([b], [[particle((1.5, 1.5, 1.5), (8 + 16 * k, 8, 8)) for k in range(n)]], max_semi=2)
    if ok:
        assert len(np.unique(sim.field("solid"))) == 1 + n
    else:
        with pytest.raises(L.LBError, match="LB_ECAPACITY"):
            sim.field("rho")
