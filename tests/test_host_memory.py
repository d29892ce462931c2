"""Host memory that runs out while a solver is assembled: no exception crosses the C interface and
none ends the process.  The coarse solves' host plans are run with failing allocations on the CPU;
cgp_assemble on the GPU, with operator new replaced by one that fails at a chosen call."""

import os
import subprocess
import sys

import pytest

from test_onchip_plan import NVCC, ROOT

CSRC = os.path.join(ROOT, "paper_1812_00185_gb300", "csrc")


def test_plan_passes_on_bad_alloc(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "check")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(NVCC))), "include")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-pthread", "-I" + include, "-o", exe, "-x", "c++",
                           os.path.join(ROOT, "tests", "host_plan_alloc_check.cpp"), os.path.join(CSRC, "rr_plan.cu")])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, (out.returncode, out.stdout, out.stderr)


NEW = r"""
#include <cstdlib>
#include <new>
static thread_local long left = 0;   // 0: not armed
extern "C" void fail_after(long k) { left = k; }
extern "C" long still_armed() { return left; }
void* operator new(size_t n) {
    if (left > 0 && --left == 0) throw std::bad_alloc();
    if (void* p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }
"""

SCRIPT = r"""
import ctypes, sys
hook = ctypes.CDLL(sys.argv[1], ctypes.RTLD_GLOBAL)   # before any library that uses operator new
sys.path.insert(0, sys.argv[2])
import numpy as np, torch
from paper_1812_00185_gb300 import binding as cg
from workloads import square_mesh
hook.still_armed.restype = ctypes.c_long
ends = set()
for n, levels, kw in ((20, 0, {}), (24, 1, {}), (64, 0, {"guess": cg.CGP_GUESS_LEARNED}), (16, 1, {"precision": cg.CGP_MIXED})):
    b = square_mesh(n)
    m = cg.Mesh(b.xy, b.tri, b.tag, levels)
    prm = cg.make_params(100.0, 0.01, k=0, **kw)
    space = torch.empty(cg.cgp_workspace_size(m.handle, prm), dtype=torch.uint8, device="cuda")
    for k in list(range(1, 30)) + [60, 200, 1000, 10 ** 9]:
        s = ctypes.c_void_p()
        hook.fail_after(ctypes.c_long(k))
        rc = cg.load().cgp_assemble(m.handle, ctypes.byref(prm), cg._ptr(space), ctypes.c_size_t(space.numel()),
                                    cg._stream(None), ctypes.byref(s))
        hook.fail_after(ctypes.c_long(0))
        assert rc in (cg.CGP_OK, cg.CGP_ENOMEM), rc
        assert (rc == cg.CGP_OK) == bool(s.value)
        ends.add(rc)
        if s.value:
            rhs = np.random.default_rng(k).standard_normal(cg.cgp_solver_info(s)[1])
            phi, it, rc = cg.cgp_poisson_solve(s, rhs - rhs.mean())
            assert rc == cg.CGP_OK and np.isfinite(phi).all()
            cg.cgp_solver_destroy(s)
    m.close()
assert ends == {cg.CGP_OK, cg.CGP_ENOMEM}, ends
print("done")
"""


@pytest.mark.gpu
def test_assembly_survives_bad_alloc(lib, tmp_path):
    src, so = str(tmp_path / "new.cpp"), str(tmp_path / "new.so")
    with open(src, "w") as f:
        f.write(NEW)
    subprocess.check_call(["g++", "-O2", "-shared", "-fPIC", "-o", so, src])
    out = subprocess.run([sys.executable, "-c", SCRIPT, so, ROOT], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and "done" in out.stdout, (out.returncode, out.stdout, out.stderr[-2000:])
