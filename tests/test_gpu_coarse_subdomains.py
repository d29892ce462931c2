"""The register-resident FP64 solve over compact subdomains (rr_plan.cuh), which the learned guess
takes: clusters of 8 and of 4 CTAs, ragged last CTAs, prescribed values, a start that is not zero,
and steps in which the network's start is taken or left.  The criteria are the solve's own contract
(as in test_gpu_coarse_grid.py) and, over steps, the fields of the solver without the network."""

import numpy as np
import pytest

from test_gpu_coarse_grid import TOL, _rhs, _system
from workloads import channel_cylinder_mesh, square_mesh

pytestmark = pytest.mark.gpu

# (base mesh, levels): 4,225 rows to 66,049 and about 68,000, which take clusters of 4
CASES = {
    "sq64": lambda: (square_mesh(64), 0), "sq129": lambda: (square_mesh(129), 0), "sq64_l1": lambda: (square_mesh(64), 1),
    "channel": lambda: (channel_cylinder_mesh(seed=3, h=0.012), 0), "channel_l1": lambda: (channel_cylinder_mesh(seed=3, h=0.012), 1),
    "sq256": lambda: (square_mesh(256), 0), "channel_l2": lambda: (channel_cylinder_mesh(seed=3, h=0.0116), 2),
}


@pytest.mark.parametrize("name", CASES)
def test_subdomain_solve_meets_its_tolerance(lib, name):
    from paper_1812_00185_gb300 import binding as cg
    base, levels = CASES[name]()
    m, s, A, fixed = _system(cg, base, levels)
    s.close()
    s = cg.Solver(m, cg.make_params(100.0, 0.01, k=0, guess=cg.CGP_GUESS_LEARNED, tol_poisson=TOL, max_it_poisson=20000))
    kind, ctas, _ = s.coarse_info()
    assert kind == cg.CGP_COARSE_PERSISTENT and s.coarse_subdomains() == ctas > 16
    plain = cg.Solver(m, cg.make_params(100.0, 0.01, k=0, guess=cg.CGP_GUESS_ZERO, tol_poisson=TOL, max_it_poisson=20000,
                                        precond=cg.CGP_PRECOND_JACOBI))
    b = _rhs(A.shape[0], fixed, 17)
    first, it, rc = cg.cgp_poisson_solve(s.handle, b)
    again = cg.cgp_poisson_solve(s.handle, b)[0]
    assert rc == cg.CGP_OK and np.array_equal(first, again)
    assert np.linalg.norm(b - A @ first) <= 1.01 * TOL * np.linalg.norm(b)
    assert 0 < it < cg.cgp_poisson_solve(plain.handle, b)[1]
    plain.close()
    # prescribed values and a start
    g = np.random.default_rng(18)
    b, start = g.standard_normal(A.shape[0]), g.standard_normal(A.shape[0])
    b = b if fixed.any() else b - b.mean()
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b, start)
    assert rc == cg.CGP_OK and np.linalg.norm(b - A @ phi) <= 1.01 * TOL * np.linalg.norm(b)
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b, phi)
    assert rc == cg.CGP_OK and it == 0
    s.close()
    m.close()


def _damped_jacobi(rms):
    """Weights of a network that predicts q + rms(q) c r / rms(r), c = 0.05 rms: in the first step
    (q = 0, whose scale is 1) 0.05 b, which lowers the residual of the zero start."""
    W1, W2, W3 = np.zeros((64, 8)), np.zeros((64, 128)), np.zeros(128)
    W1[0, 0], W1[1, 0], W2[0, 0], W2[1, 1], W3[0], W3[1] = 1.0, -1.0, 1.0, 1.0, 0.05 * rms, -0.05 * rms
    z = np.zeros(64)
    return np.concatenate([W1.ravel(), z, W2.ravel(), z, W3, [0.0]]).astype(np.float32)


@pytest.mark.parametrize("network", ["jacobi", "noise"])
def test_steps_with_a_second_start(lib, network):
    from paper_1812_00185_gb300 import binding as cg
    from paper_1812_00185_gb300.learned import init_params
    common = dict(chi=1, k=1, bc_kind=cg.CGP_BC_CHANNEL, bc_param=(0.3, 0.41), tol_mom=1e-11, tol_poisson=1e-10,
                  tol_mass=1e-11)
    base = channel_cylinder_mesh(seed=11, h=0.022)
    m = cg.Mesh(base.xy, base.tri, base.tag, 2)
    net = cg.cgp_mlp_create(m.handle, 1, 1)
    out = {}
    for guess in (cg.CGP_GUESS_PROJ, cg.CGP_GUESS_LEARNED):
        s = cg.Solver(m, cg.make_params(1000.0, 0.002, guess=guess, **common))
        if guess == cg.CGP_GUESS_LEARNED:
            if network == "jacobi":
                p = _damped_jacobi(rms)
            else:
                p = init_params(5)
                p[p.size - 129:p.size - 1] *= 1000.0
            cg.cgp_mlp_set_params(net, p)
            cg.cgp_guess_set(s.handle, net)
            assert s.coarse_info()[0] == cg.CGP_COARSE_PERSISTENT and s.coarse_subdomains() > 16
        s.step(1)
        rms = float(np.sqrt(np.mean(s.vector(cg.CGP_VEC_RHS_C) ** 2)))
        first = s.fields()[3]["guess_used"]
        s.step(29)
        U, P, t, st, rc = s.fields()
        assert rc == cg.CGP_OK and st["res_poisson"] <= 1.0001e-10
        out[guess] = U, P, first
        s.close()
    assert out[cg.CGP_GUESS_LEARNED][2] == (1 if network == "jacobi" else 0)
    for a, b in zip(out[cg.CGP_GUESS_LEARNED][:2], out[cg.CGP_GUESS_PROJ][:2]):
        assert np.linalg.norm(a - b) / np.linalg.norm(b) < 1e-6
    cg.cgp_mlp_destroy(net)
    m.close()
