"""Which caller memory the warm start's kernels use in place (in_place_view in lbsph_internal.cuh), on the host with made-up
pointer attributes: the context GPU's own memory, managed and page-locked memory.  An array of another GPU of the process,
which a copy reaches without peer access and a kernel does not, pageable memory and a range over two mappings must go
through a copy, and both calls that take device arrays must ask."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2403_05443_gb300", "csrc")

PROG = r"""
#include "lbsph_internal.cuh"
#include <cstdio>
using namespace lbsph;
static cudaPointerAttributes at(cudaMemoryType t, int dev, unsigned long long p) {
    cudaPointerAttributes a{};
    a.type = t;
    a.device = dev;
    a.devicePointer = reinterpret_cast<void*>(p);
    return a;
}
static int bad = 0;
static void expect(const char* what, const cudaPointerAttributes& a, const cudaPointerAttributes& b, size_t n, int dev, bool yes) {
    void* want = yes ? a.devicePointer : nullptr;
    if (in_place_view(a, b, n, dev) != want) { printf("%s\n", what); ++bad; }
}
int main() {
    const unsigned long long P = 0x7f0000000000ull;
    const size_t n = 12 << 20;
    const auto D = cudaMemoryTypeDevice, M = cudaMemoryTypeManaged, H = cudaMemoryTypeHost, U = cudaMemoryTypeUnregistered;
    expect("own device memory", at(D, 0, P), at(D, 0, P + n - 1), n, 0, true);
    expect("own memory of device 1", at(D, 1, P), at(D, 1, P + n - 1), n, 1, true);
    expect("another GPU's memory", at(D, 1, P), at(D, 1, P + n - 1), n, 0, false);
    expect("managed", at(M, 1, P), at(M, 1, P + n - 1), n, 0, true);
    expect("page-locked", at(H, 0, P), at(H, 0, P + n - 1), n, 0, true);
    expect("pageable", at(U, -2, 0), at(U, -2, 0), n, 0, false);
    expect("end beyond the mapping", at(D, 0, P), at(U, -2, 0), n, 0, false);
    expect("two mappings", at(D, 0, P), at(D, 0, P + 2 * n), n, 0, false);
    printf("%s\n", bad ? "FAIL" : "OK");
    return bad != 0;
}
"""


def test_only_memory_that_the_gpu_reaches_is_used_in_place(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "view.cu", tmp_path / "view"
    src.write_text(PROG)
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-I", SRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout


@pytest.mark.parametrize("call,args", [("lb_init_fluid", ("u", "drho")), ("lb_stokes_field", ("u_dev", "drho_dev"))])
def test_the_warm_start_asks_for_every_device_array(call, args):
    with open(os.path.join(SRC, "lbsph_api.cu")) as f:
        text = f.read()
    body = re.search(r'extern "C" lb_status %s\(.*?\n}\n' % call, text, re.S).group(0)
    for a in args:
        assert re.search(r"device_view\(ctx, %s," % a, body), a
