"""The FP64 coarse solve with the matrix's inverse: from three rows to the largest system it takes,
whole and ragged slices, prescribed values, a zero right-hand side, a start that is not zero, and
the systems and caps that stay with PCG.  The criterion is the solve's own contract, checked on the
host as in test_gpu_coarse_grid.py."""

import numpy as np
import pytest
from scipy.sparse.csgraph import connected_components

from test_gpu_coarse_grid import TOL, _fan, _rhs, _system
from workloads import channel_cylinder_mesh, square_mesh

pytestmark = pytest.mark.gpu

CASES = {
    "sq1": lambda: (square_mesh(1), 0), "fan31": lambda: (_fan(31), 0), "fan32": lambda: (_fan(32), 0),
    "sq5_l2": lambda: (square_mesh(5), 2), "sq39": lambda: (square_mesh(39), 0),
    "channel": lambda: (channel_cylinder_mesh(seed=4, h=0.03), 0), "channel_l1": lambda: (channel_cylinder_mesh(seed=4, h=0.05), 1),
}


@pytest.mark.parametrize("name", CASES)
def test_direct_solve_meets_its_tolerance(lib, name):
    from paper_1812_00185_gb300 import binding as cg
    base, levels = CASES[name]()
    m, s, A, fixed = _system(cg, base, levels)
    b = _rhs(A.shape[0], fixed, 21)
    out = []
    for _ in range(2):
        phi, it, rc = cg.cgp_poisson_solve(s.handle, b)
        assert rc == cg.CGP_OK and 1 <= it <= 3
        assert np.linalg.norm(b - A @ phi) <= 1.01 * TOL * np.linalg.norm(b)
        out.append(phi)
    assert np.array_equal(out[0], out[1])
    phi, it, rc = cg.cgp_poisson_solve(s.handle, np.zeros_like(b), out[0])
    assert rc == cg.CGP_OK and it == 0 and not phi.any()
    s.close()
    m.close()


def test_direct_solve_with_prescribed_values_and_a_start(lib):
    from paper_1812_00185_gb300 import binding as cg
    m, s, A, fixed = _system(cg, channel_cylinder_mesh(seed=4, h=0.05), 1)
    s.close()
    s = cg.Solver(m, cg.make_params(100.0, 0.01, k=0, tol_poisson=TOL, max_it_poisson=20000))
    g = np.random.default_rng(22)
    b, start = g.standard_normal(A.shape[0]), g.standard_normal(A.shape[0])
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b, start)
    assert rc == cg.CGP_OK and it >= 1
    assert np.linalg.norm(b - A @ phi) <= 1.01 * TOL * np.linalg.norm(b)
    again, it, rc = cg.cgp_poisson_solve(s.handle, b, phi)
    assert rc == cg.CGP_OK and it == 0 and np.array_equal(again, phi)
    s.close()
    m.close()


@pytest.mark.parametrize("n,cap", [(16, 63), (40, 20000)])
def test_small_caps_and_larger_systems_stay_iterative(lib, n, cap):
    # a cap below 64 is one on PCG iterations; 41^2 rows are beyond the inverse
    from paper_1812_00185_gb300 import binding as cg
    m = cg.Mesh(square_mesh(n).xy, square_mesh(n).tri, square_mesh(n).tag, 0)
    s = cg.Solver(m, cg.make_params(100.0, 0.01, k=0, guess=cg.CGP_GUESS_ZERO, tol_poisson=TOL, max_it_poisson=cap))
    b = _rhs((n + 1) ** 2, np.zeros((n + 1) ** 2, bool), 23)
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b)
    assert it > 10 and np.isfinite(phi).all() and (rc == cg.CGP_OK or it >= cap)
    s.close()
    m.close()


def test_two_part_mesh_stays_iterative(lib):
    from paper_1812_00185_gb300 import binding as cg
    a = square_mesh(12)
    both = type("Base", (), {"xy": np.concatenate([a.xy, a.xy + [2.0, 0.0]]),
                             "tri": np.concatenate([a.tri, a.tri + len(a.xy)]).astype(np.int32),
                             "tag": np.concatenate([a.tag, a.tag])})
    m, s, A, fixed = _system(cg, both, 0)
    part = connected_components(A)[1]
    b = np.random.default_rng(24).standard_normal(A.shape[0])
    for p in (0, 1):
        b[part == p] -= b[part == p].mean()
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b)
    assert rc == cg.CGP_OK and it > 3 and np.linalg.norm(b - A @ phi) <= 1.01 * TOL * np.linalg.norm(b)
    s.close()
    m.close()
