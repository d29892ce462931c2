"""The multilevel solve on a large base mesh alone (more than 20 slices per CTA: 32 warps a CTA and
8 of them per subdomain), pure Neumann and with prescribed values on three sides: the solve's own
contract, as in test_gpu_coarse_grid.py, and the same bits twice."""

import numpy as np
import pytest

from test_gpu_coarse_grid import TOL, _rhs, _system
from workloads import square_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,fixed_sides", [(330, False), (330, True), (420, True)])
def test_large_base_mesh_solve_meets_its_tolerance(lib, n, fixed_sides):
    from paper_1812_00185_gb300 import binding as cg
    base = square_mesh(n)
    if fixed_sides:
        x, y = base.xy.T
        base.tag[(x == 0) | (x == 1) | (y == 1)] |= cg.CGP_PHI_ZERO
    m, s, A, fixed = _system(cg, base, 0)
    assert fixed.any() == fixed_sides and A.shape[0] > 20 * 32 * s.coarse_info()[1] and A.shape[0] % 32
    assert s.coarse_info()[0] == cg.CGP_COARSE_PERSISTENT_MEM and s.coarse_subdomains() == 4 * s.coarse_info()[1]
    b = _rhs(A.shape[0], fixed, 15)
    first, it, rc = cg.cgp_poisson_solve(s.handle, b)
    assert rc == cg.CGP_OK and 0 < it < 700
    assert np.linalg.norm(b - A @ first) <= 1.01 * TOL * np.linalg.norm(b)
    assert np.array_equal(cg.cgp_poisson_solve(s.handle, b)[0], first)
    # prescribed values and a start that is not zero
    s.close()
    s = cg.Solver(m, cg.make_params(100.0, 0.01, k=0, tol_poisson=TOL, max_it_poisson=20000))
    g = np.random.default_rng(16)
    b, start = g.standard_normal(A.shape[0]), g.standard_normal(A.shape[0])
    b = b if fixed_sides else b - b.mean()
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b, start)
    assert rc == cg.CGP_OK and np.array_equal(phi[fixed], b[fixed])
    assert np.linalg.norm(b - A @ phi) <= 1.01 * TOL * np.linalg.norm(b)
    s.close()
    m.close()
