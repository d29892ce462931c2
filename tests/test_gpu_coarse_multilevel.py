"""The multilevel FP64 coarse solve at the edges of its range: base meshes smaller and larger than
the subdomains, one to four levels below, few and many slices per CTA (stored and recomputed
prolongations), a warp or 8 warps per subdomain, prescribed values and a start that is not zero.
The criterion is the solve's own contract, checked on the host as in test_gpu_coarse_grid.py."""

import numpy as np
import pytest
from scipy.sparse.csgraph import connected_components

from test_gpu_coarse_grid import TOL, _fan, _rhs, _system
from workloads import channel_cylinder_mesh, square_mesh

pytestmark = pytest.mark.gpu

# (base mesh, levels below): 4,097 rows and more; beyond 155,648 (32 slices per CTA) z is stored
CASES = {
    "fan32_l4": lambda: (_fan(32), 4), "sq4_l4": lambda: (square_mesh(4), 4), "sq32_l1": lambda: (square_mesh(32), 1),
    "sq13_l3": lambda: (square_mesh(13), 3), "channel_l2": lambda: (channel_cylinder_mesh(seed=3, h=0.03), 2),
    "sq36_l4": lambda: (square_mesh(36), 4), "sq90_l2": lambda: (square_mesh(90), 2), "sq200_l1": lambda: (square_mesh(200), 1),
    "sq100_l2": lambda: (square_mesh(100), 2), "sq50_l3": lambda: (square_mesh(50), 3),
    "channel_l4": lambda: (channel_cylinder_mesh(seed=3, h=0.03), 4),
}


@pytest.mark.parametrize("name", CASES)
def test_multilevel_solve_meets_its_tolerance(lib, name):
    from paper_1812_00185_gb300 import binding as cg
    base, levels = CASES[name]()
    m, s, A, fixed = _system(cg, base, levels)
    n0 = len(base.xy)
    assert s.coarse_info()[0] == cg.CGP_COARSE_PERSISTENT_MEM and s.coarse_subdomains() == min(n0, 4 * s.coarse_info()[1])
    b = _rhs(A.shape[0], fixed, 11)
    for _ in range(2):      # the second pass on the same solver gives the same bits
        phi, it, rc = cg.cgp_poisson_solve(s.handle, b)
        assert rc == cg.CGP_OK and 0 < it < 250
        assert np.linalg.norm(b - A @ phi) <= 1.01 * TOL * np.linalg.norm(b)
        first = phi if _ == 0 else first
    assert np.array_equal(phi, first)
    s.close()
    m.close()


def test_multilevel_solve_with_prescribed_values_and_a_start(lib):
    # b at phi = 0 rows is their solution (identity rows); the solve starts from the given phi
    from paper_1812_00185_gb300 import binding as cg
    base = channel_cylinder_mesh(seed=3, h=0.03)
    m, s, A, fixed = _system(cg, base, 2)
    s.close()
    s = cg.Solver(m, cg.make_params(100.0, 0.01, k=0, tol_poisson=TOL, max_it_poisson=20000))
    g = np.random.default_rng(12)
    b, start = g.standard_normal(A.shape[0]), g.standard_normal(A.shape[0])
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b, start)
    assert rc == cg.CGP_OK and it > 0
    assert np.array_equal(phi[fixed], b[fixed])
    assert np.linalg.norm(b - A @ phi) <= 1.01 * TOL * np.linalg.norm(b)
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b, phi)     # solved already: nothing to do
    assert rc == cg.CGP_OK and it == 0
    s.close()
    m.close()


def test_two_part_mesh_falls_back_to_jacobi(lib):
    # constants on either part: the base mesh's coarse matrix is singular beyond the constants
    from paper_1812_00185_gb300 import binding as cg
    a = square_mesh(24)
    both = type("Base", (), {"xy": np.concatenate([a.xy, a.xy + [2.0, 0.0]]),
                             "tri": np.concatenate([a.tri, a.tri + len(a.xy)]).astype(np.int32),
                             "tag": np.concatenate([a.tag, a.tag])})
    m, s, A, fixed = _system(cg, both, 1)
    assert s.coarse_subdomains() == 0
    n = A.shape[0]
    part = connected_components(A)[1]
    b = np.random.default_rng(13).standard_normal(n)
    for p in (0, 1):
        b[part == p] -= b[part == p].mean()
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b)
    assert rc == cg.CGP_OK and np.linalg.norm(b - A @ phi) <= 1.01 * TOL * np.linalg.norm(b)
    s.close()
    m.close()


# the base mesh itself: M^{-1} = D^{-1} + Z E^+ Z^T, a warp or 8 warps per subdomain
FLAT = {"sq40": lambda: square_mesh(40), "channel": lambda: channel_cylinder_mesh(seed=3, h=0.012),
        "sq64": lambda: square_mesh(64), "sq197": lambda: square_mesh(197)}


@pytest.mark.parametrize("name", FLAT)
def test_base_mesh_solve_meets_its_tolerance(lib, name):
    from paper_1812_00185_gb300 import binding as cg
    m, s, A, fixed = _system(cg, FLAT[name](), 0)
    assert s.coarse_info()[0] == cg.CGP_COARSE_PERSISTENT_MEM and s.coarse_subdomains() == 4 * s.coarse_info()[1]
    b = _rhs(A.shape[0], fixed, 14)
    first = cg.cgp_poisson_solve(s.handle, b)
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b)
    assert rc == cg.CGP_OK and 0 < it < 400 and np.array_equal(phi, first[0])
    assert np.linalg.norm(b - A @ phi) <= 1.01 * TOL * np.linalg.norm(b)
    s.close()
    m.close()
