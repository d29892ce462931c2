"""FP64 coarse solves of very small and very large loads.  A load times a power of two has the same
solve, bit for bit, times that power (nothing in it overflows or underflows at 2^400 times loads of
ordinary size), in every kernel; and the kernels' quotient by Newton's iteration agrees with / from
the smallest to the largest divisors."""

import os
import subprocess

import numpy as np
import pytest

from test_gpu_coarse_grid import TOL, _rhs
from test_onchip_plan import NVCC, ROOT
from workloads import channel_cylinder_mesh, square_mesh

pytestmark = pytest.mark.gpu

CASES = {   # mesh, levels, preconditioner, coarse solver
    "one_cluster": (square_mesh, 40, 0, "JACOBI", "PERSISTENT"), "clusters": (square_mesh, 150, 0, "JACOBI", "PERSISTENT"),
    "memory": (square_mesh, 48, 0, "JACOBI", "PERSISTENT_MEM"), "cluster": (square_mesh, 48, 0, "JACOBI", "CLUSTER"),
    "inverse": (square_mesh, 30, 0, "AUTO", "AUTO"), "multilevel": (square_mesh, 24, 2, "AUTO", "AUTO"),
    "base_mesh": (square_mesh, 60, 0, "AUTO", "AUTO"), "channel": (channel_cylinder_mesh, 0.03, 1, "JACOBI", "PERSISTENT"),
    "channel_multilevel": (channel_cylinder_mesh, 0.03, 1, "AUTO", "AUTO"),
}


@pytest.mark.parametrize("name", CASES)
def test_scaled_loads_have_scaled_solutions(lib, name):
    from paper_1812_00185_gb300 import binding as cg
    make, size, levels, precond, mode = CASES[name]
    base = make(seed=2, h=size) if make is channel_cylinder_mesh else make(size)
    m = cg.Mesh(base.xy, base.tri, base.tag, levels)
    s = cg.Solver(m, cg.make_params(100.0, 0.01, k=0, guess=cg.CGP_GUESS_ZERO, tol_poisson=TOL, max_it_poisson=20000,
                                    precond=getattr(cg, "CGP_PRECOND_" + precond),
                                    coarse_mode=getattr(cg, "CGP_COARSE_" + mode)))
    b = _rhs(s.nc, (m.level(levels)["tag"] & cg.CGP_PHI_ZERO) != 0, 31)
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b)
    assert rc == cg.CGP_OK
    for p in (-400, 400):
        got, it2, rc = cg.cgp_poisson_solve(s.handle, np.ldexp(b, p))
        assert rc == cg.CGP_OK and it2 == it and np.array_equal(got, np.ldexp(phi, p)), (p, it2, it)
    s.close()
    m.close()


def test_newton_quotient_agrees_with_division(lib, tmp_path):
    # two steps from 20 bits leave 2^-80; two roundings of the quotient: 2^-52 of the exact one,
    # which n / d itself rounds to within 2^-53
    exe, src, dst = str(tmp_path / "check"), str(tmp_path / "in"), str(tmp_path / "out")
    subprocess.check_call([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17",
                           "-I" + os.path.join(ROOT, "include"), "-o", exe, os.path.join(ROOT, "tests", "newton_quotient_check.cu")])
    g = np.random.default_rng(6)
    e = np.repeat(np.arange(-1074, 1024), 64)             # every exponent, subnormal ones too
    d = np.ldexp(g.uniform(1.0, 2.0, e.size), e) * g.choice([-1.0, 1.0], e.size)
    q = np.ldexp(g.uniform(1.0, 2.0, e.size), g.integers(-20, 20, e.size))
    with np.errstate(over="ignore", under="ignore"):
        n = d * q
        ok = np.isfinite(n) & (np.abs(n) >= 2.0 ** -1022)   # a normal numerator and quotient
        n, d = n[ok], d[ok]
        want = n / d
    keep = np.isfinite(want) & (np.abs(want) >= 2.0 ** -1000)
    n, d, want = n[keep], d[keep], want[keep]
    bad = np.array([0.0, -0.0, np.inf, -np.inf, np.nan])
    np.concatenate([n, np.ones(5), d, bad]).tofile(src)
    subprocess.check_call([exe, str(n.size + 5), src, dst])
    got = np.fromfile(dst)
    assert np.abs(got[:-5] / want - 1.0).max() <= 2.0 ** -52 + 2.0 ** -53
    assert not np.isfinite(got[-5:]).any()
    assert (np.abs(d) < 2.0 ** -1022).any() and (np.abs(d) >= 2.0 ** 1022).any()
