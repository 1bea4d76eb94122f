"""Field read-back: density, velocity, populations and owner field of one state belong together.

The nodes next to a surface and all others are done by different blocks (one thread per cube node, one per four x
nodes); both must give the moments of the populations they give, and zeros inside.  Cubes across every face of the
box, partners that share nodes, walls, squirmers, rows shorter and longer than a warp, 16-bit storage, and the state
before the first step."""
import numpy as np
import pytest

from lb_inputs import box, particle, random_quaternion, rng

pytestmark = pytest.mark.gpu

L = pytest.importorskip("paper_2403_05443_gb300.lbsph")

CASES = {
    "corner": (box(24, 20, 22, 0.8, counter_force=1),
               [dict(semi=(4.5, 2.5, 2.0), c=(0.2, 19.7, 0.4), U=(0.03, 0.02, -0.03), F_ext=(1e-3, 0, 0))]),
    "partners": (box(40, 32, 32, 0.9, counter_force=1),
                 [dict(semi=(3.5, 3.5, 3.5), c=(14.3, 15.8, 16.1), U=(0.02, 0, 0), F_ext=(3e-3, 0, 0)),
                  dict(semi=(4.5, 2.5, 2.0), c=(23.15, 16.2, 15.9), U=(-0.02, 0.01, 0), B1=1e-3, B2=2e-3)]),
    "walls": (box(136, 24, 20, 1.0, walls=1, wall_u_lo=(-0.01, 0, 0), wall_u_hi=(0.01, 0, 0.002)),
              [dict(semi=(5.0, 2.5, 2.5), c=(134.9, 11.3, 0.6), U=(0.03, 0, 0.02))]),
    "empty": (box(24, 16, 18, 1.1, body_force=(1e-5, 0, -2e-5)), []),
}


@pytest.mark.parametrize("steps", [0, 1, 17])
@pytest.mark.parametrize("prec", [L.LB_FP32, L.LB_FP16, L.LB_BF16])
@pytest.mark.parametrize("name", CASES)
def test_readback_fields_belong_together(name, prec, steps):
    b, ps = CASES[name]
    g = rng(77)
    parts = [particle(p["semi"], p["c"], random_quaternion(g), **{k: v for k, v in p.items() if k not in ("semi", "c")})
             for p in ps]
    sim = L.Simulation([b], [parts], precision=prec, max_semi=5)
    sim.step(steps)
    df, f = sim.field("df").astype(np.float64), sim.field("f").astype(np.float64)
    rho, u, own = sim.field("rho").astype(np.float64), sim.field("u").astype(np.float64), sim.field("solid")
    c, w = L.lb_lattice()
    c, w = np.asarray(c, float), np.asarray(w, float)
    fluid = own == 0
    assert (df[:, ~fluid] == 0).all() and (rho.reshape(fluid.shape)[~fluid] == 0).all() and (u[:, ~fluid] == 0).all()
    # full populations: one FP32 rounding of df + w rho0 <= 1/3 + small
    assert np.abs(f - (df + w[:, None, None, None]))[:, fluid].max() <= 2.0 ** -24
    # a sum of 19 FP32 numbers: at most 18 roundings of partial sums <= sum |f|
    eps = 2.0 ** -24
    size = np.abs(df).sum(0)[fluid]
    assert (np.abs(rho.reshape(fluid.shape)[fluid] - df.sum(0)[fluid]) <= 18 * eps * size).all()
    # velocity: ten differences, the half force and the division by rho0 + drho (|u| well below 1)
    gbox = np.array(b.get("body_force", (0, 0, 0)), float)
    if b.get("counter_force"):
        gbox = gbox - sum(np.array(p.get("F_ext", (0, 0, 0)), float) for p in parts) / fluid.sum()
    j = np.einsum("ia,ikyx->akyx", c, df)[:, fluid] + 0.5 * gbox[:, None]
    ref = j / (1.0 + df.sum(0)[fluid])
    assert (np.abs(u[:, fluid] - ref) <= 24 * eps * (size + np.abs(gbox).max() + np.abs(ref))).all()
