"""lb_get_force_torque for many particles at once: the records of all of them (gathered with one double per thread, so
256 to a block; up to 512 records into page-locked memory, above that into device memory with a copy behind it: counts
on both sides of each edge) are what lb_get_force_torque_async copies straight out of the particle states, also those
of one box in the middle.

The call's time must stay near that of such a copy: with one block for all records 4,096 of them took 137 us, the copy
with its wait 31.  Bar 3 (medians of 41 in turn): the gathering and the status word may cost as much again."""
import time

import numpy as np
import pytest

from lb_inputs import box, particle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
L = pytest.importorskip("paper_2403_05443_gb300.lbsph")


def _sim(n):
    """n unit spheres, up to 64 to a box of 64^3."""
    sites = [(8 + 16 * i, 8 + 16 * j, 8 + 16 * k) for k in range(4) for j in range(4) for i in range(4)]
    left, parts = n, []
    while left > 0:
        parts.append([particle((1, 1, 1), s, F_ext=(1e-4 * (1 + len(parts)), 1e-5 * k, 0)) for k, s in enumerate(sites[:left])])
        left -= len(parts[-1])
    sim = L.Simulation([box(64, 64, 64, 1.0)] * len(parts), parts, max_semi=1, precision=L.LB_BF16)
    sim.step(3)
    return sim


@pytest.mark.parametrize("n", [1, 10, 11, 512, 513, 1024])
def test_records_of_many_particles(n):
    sim = _sim(n)
    out = np.full((n, L.LB_RECORD_DOUBLES), np.nan)
    L.lb_get_force_torque(sim.ctx, -1, n, out)
    dev = torch.zeros((n, L.LB_RECORD_DOUBLES), dtype=torch.float64, device="cuda")
    L.lb_get_force_torque_async(sim.ctx, -1, n, dev.data_ptr())
    sim.sync()
    assert np.array_equal(out, dev.cpu().numpy()) and (out[:, 12] > 0).all()
    b = len(sim.boxes) // 2
    assert np.array_equal(sim.records(b), out[64 * b:64 * b + sim.nparts[b]])


def test_call_takes_about_as_long_as_a_copy():
    n = 4096
    sim = _sim(n)
    out = np.zeros((n, L.LB_RECORD_DOUBLES))
    s = torch.cuda.Stream()
    t = {"call": [], "copy": []}
    for _ in range(45):
        a = time.perf_counter()
        L.lb_get_force_torque(sim.ctx, -1, n, out)
        b = time.perf_counter()
        L.lb_get_force_torque_async(sim.ctx, -1, n, out.ctypes.data, s.cuda_stream)
        s.synchronize()
        t["call"].append(b - a)
        t["copy"].append(time.perf_counter() - b)
    m = {k: float(np.median(v[4:])) for k, v in t.items()}
    assert m["call"] <= 3 * m["copy"], m
