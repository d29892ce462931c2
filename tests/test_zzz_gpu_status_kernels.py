"""The statuses of test_zzz_gpu_status.py in each of the FP64 coarse kernels (no GPU fault, trap or
hang): a NaN right-hand side, and a bounded device wait that runs out under the cgp_set_wait_test
hook.  The register-resident solve on one cluster and on clusters of 8 and of 4 CTAs (word polls,
mbarriers), the same with its subdomain plan, the multilevel solve with and without a level below,
the memory-resident grid solve (grid barriers), and one cluster (NaN alone: hardware barriers)."""

import time

import numpy as np
import pytest

from workloads import channel_cylinder_mesh, square_mesh

pytestmark = pytest.mark.gpu

CASES = {   # base mesh, levels, parameters, (kind, subdomains or not, CTAs at least)
    "one_cluster": (lambda: square_mesh(40), 0, {"precond": "JACOBI"}, ("PERSISTENT", False, 16)),
    "clusters_of_8": (lambda: square_mesh(129), 0, {"precond": "JACOBI"}, ("PERSISTENT", False, 17)),
    "clusters_dirichlet": (lambda: channel_cylinder_mesh(seed=4, h=0.03), 2, {"precond": "JACOBI"}, ("PERSISTENT", False, 17)),
    "clusters_of_4": (lambda: square_mesh(256), 0, {"precond": "JACOBI"}, ("PERSISTENT", False, 100)),
    "subdomains": (lambda: square_mesh(129), 0, {"guess": "LEARNED"}, ("PERSISTENT", True, 17)),
    "multilevel": (lambda: square_mesh(32), 2, {}, ("PERSISTENT_MEM", True, 17)),
    "multilevel_dirichlet": (lambda: channel_cylinder_mesh(seed=4, h=0.03), 1, {}, ("PERSISTENT_MEM", True, 17)),
    "base_mesh": (lambda: square_mesh(64), 0, {}, ("PERSISTENT_MEM", True, 17)),
    "memory": (lambda: square_mesh(64), 0, {"precond": "JACOBI", "coarse_mode": "PERSISTENT_MEM"}, ("PERSISTENT_MEM", False, 2)),
    "cluster": (lambda: square_mesh(64), 0, {"precond": "JACOBI", "coarse_mode": "CLUSTER"}, ("CLUSTER", False, 2)),
}
PREFIX = {"precond": "CGP_PRECOND_", "guess": "CGP_GUESS_", "coarse_mode": "CGP_COARSE_"}


def _solver(cg, name):
    make, levels, kw, (kind, subdomains, ctas) = CASES[name]
    base = make()
    kw = {k: getattr(cg, PREFIX[k] + v) for k, v in kw.items()}
    kw.setdefault("guess", cg.CGP_GUESS_ZERO)
    m = cg.Mesh(base.xy, base.tri, base.tag, levels)
    s = cg.Solver(m, cg.make_params(100.0, 0.01, k=0, tol_poisson=1e-10, max_it_poisson=20000, **kw))
    info = s.coarse_info()
    assert info[0] == getattr(cg, "CGP_COARSE_" + kind) and info[1] >= ctas and (s.coarse_subdomains() > 0) == subdomains
    return m, s


def _converges(cg, s, r):
    phi, it, rc = cg.cgp_poisson_solve(s.handle, r)
    assert rc == cg.CGP_OK and it > 0 and np.isfinite(phi).all()
    return phi


@pytest.mark.parametrize("name", CASES)
def test_nan_rhs_reports_nonfinite_then_recovers(lib, name):
    from paper_1812_00185_gb300 import binding as cg
    m, s = _solver(cg, name)
    r = np.random.default_rng(3).standard_normal(s.nc)
    good = _converges(cg, s, r)
    for at in (slice(None, None, 3), slice(s.nc // 2, s.nc // 2 + 1)):
        bad = r.copy()
        bad[at] = np.nan
        with pytest.raises(cg.CgpError) as e:
            cg.cgp_poisson_solve(s.handle, bad)
        assert e.value.code == cg.CGP_ENONFINITE
    assert np.array_equal(_converges(cg, s, r), good)
    s.close()
    m.close()


@pytest.mark.parametrize("name", [n for n in CASES if n != "cluster"])
def test_wait_that_runs_out_reports_timeout_then_recovers(lib, name):
    from paper_1812_00185_gb300 import binding as cg
    m, s = _solver(cg, name)
    r = np.random.default_rng(5).standard_normal(s.nc)
    good = _converges(cg, s, r)
    cg.cgp_set_wait_test(s.handle, 1)
    t0 = time.time()
    with pytest.raises(cg.CgpError) as e:
        cg.cgp_poisson_solve(s.handle, r)
    assert e.value.code == cg.CGP_ETIMEOUT
    assert time.time() - t0 < 5.0          # the short limit, not the seconds-long one
    cg.cgp_set_wait_test(s.handle, 0)
    assert np.array_equal(_converges(cg, s, r), good)
    s.close()
    m.close()
