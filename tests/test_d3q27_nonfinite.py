"""A D3Q27 particle whose state stops being finite, or leaves the range of 32-bit cube origins.

The particle kernel turns a pose into the extents of the nodes that the next lattice pass visits.  On the host:
whatever the two cube origins are (those of NaN, Inf and huge centres among them), the near pass's arithmetic must stay
inside the box.  On the GPU: the call reports the failure, and the other box of the context is bit for bit what it is
in a run where nothing fails; the failure comes in the first step (one of the two slots of box terms has never been
written then) or later, with the body centred or across the low faces."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from lb_inputs import box, particle, random_quaternion, rng

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2403_05443_gb300", "csrc")

PROG = r"""
#include "q27.cuh"
#include <cstdio>
#include <limits>
using namespace lbsph::q27;
static int bad = 0;
static void check(int o_a, int o_b, int S, int L) {
    int uo, E;
    cube_union27(o_a, o_b, S, L, uo, E);
    // the near pass: X = wrapc(uo + m, L) for 0 <= m < E, one subtraction
    const bool ok = E >= S && E <= L && uo >= 0 && uo < L && uo + (E - 1) < 2 * L;
    // both cubes inside the union where they overlap or touch
    const long long d = (long long)o_b - o_a;
    const bool holds = d > 1 || d < -1 || E == (S + (d < 0 ? -d : d) < L ? S + (d < 0 ? -d : d) : L);
    if (!ok || !holds) { if (++bad < 9) printf("o %d %d S %d L %d: uo %d E %d\n", o_a, o_b, S, L, uo, E); }
}
int main() {
    const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
    const double far[] = {nan, inf, -inf, 1e300, -1e300, 1e12, -1e12, POS_MAX27, -POS_MAX27, 4294967295.5, -2147483648.0};
    const int ends[] = {2147483647, -2147483647 - 1, 2147483000, -2147483000, 536870911, -536870912 - 31};
    for (int L : {20, 24, 33, 64, 100, 128}) {
        for (int h = 3; 2 * h + 4 <= L && h <= 31; ++h) {
            const int S = 2 * h + 2;
            int o, o2;
            for (double x : far)
                if (cube_origin27(x, h, o) || o != -h) { ++bad; printf("accepted %g\n", x); }
            for (double x : {-4.0, -0.25, 0.0, 0.5 * L, L - 0.5, 3.0 * L + 0.125, 536870911.5, -536870911.5}) {
                if (!cube_origin27(x, h, o) || o != (int)floor(x) - h) { ++bad; printf("refused %g\n", x); }
                for (int d = -3; d <= 3; ++d) check(o, o + d, S, L);
                for (double y : {-4.0, 536870911.5, -536870911.5}) { cube_origin27(y, h, o2); check(o, o2, S, L); }
                for (int e : ends) { check(o, e, S, L); check(e, o, S, L); check(e, e, S, L); }
            }
        }
    }
    printf("%s\n", bad ? "FAIL" : "OK");
    return bad != 0;
}
"""


def test_extents_stay_in_the_box_for_any_origin(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "ext.cu", tmp_path / "ext"
    src.write_text(PROG)
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-I", SRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("didt_mode", [0, 2])
@pytest.mark.parametrize("before", [0, 6])
@pytest.mark.parametrize("at,component,value,status", [
    ((16.2, 15.9, 16.4), 0, float("nan"), "LB_ENAN"),
    ((0.3, 0.2, 0.6), 4, float("nan"), "LB_ENAN"),
    ((0.3, 0.2, 0.6), 2, float("inf"), "LB_ENAN"),
    ((0.3, 31.8, 0.6), 1, -1e30, "LB_ECAPACITY"),
])
def test_failed_particle_leaves_the_other_box_alone(at, component, value, status, before, didt_mode):
    L = pytest.importorskip("paper_2403_05443_gb300.lbsph")
    g = rng(3)
    boxes = [box(32, 32, 32, 0.8, counter_force=1), box(32, 24, 36, 0.9, counter_force=1)]
    parts = [[particle((4.0, 2.5, 2.5), at, random_quaternion(g), F_ext=(2e-4, 1e-4, 0))],
             [particle((4.5, 3.0, 2.5), (5.1, 12.3, 17.7), random_quaternion(g), F_ext=(3e-4, -1e-4, 2e-4))]]

    def run(fail):
        sim = L.Simulation(boxes, parts, max_semi=5, lattice=27, didt_mode=didt_mode)
        sim.step(before)
        if fail:
            ft = np.zeros((1, 6))
            ft[0, component] = value
            sim.set_external(0, ft)
        sim.step(24)
        out = []
        if fail:
            with pytest.raises(L.LBError) as e:
                sim.records(1)
            assert str(e.value).startswith(status)
        for name, shape in (("df", (27,)), ("rho", ()), ("u", (3,)), ("solid", ())):
            a = np.zeros(shape + (36, 24, 32), np.float32)
            try:
                L.lb_get_fields(sim.ctx, 1, L._FIELD_NAMES[name], a.ctypes.data, a.nbytes, False)
            except L.LBError:
                assert fail
            out.append(a)
        rec = np.zeros((1, L.LB_RECORD_DOUBLES))
        L.library().lb_get_force_torque(sim.ctx, 1, rec.ctypes.data_as(L.C.POINTER(L.C.c_double)), 1)
        return out + [rec]

    for a, b in zip(run(True), run(False)):
        assert np.array_equal(a, b) and np.isfinite(a.view(np.float32) if a.dtype == np.float32 else a).all() and a.any()
