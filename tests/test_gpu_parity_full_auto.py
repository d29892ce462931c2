"""GPU parity at the benchmarked sizes with the library's FP64 default: the coarse solve's
preconditioner left to the library (the named FP64 forms ask for Jacobi alone).  Steps replayed as
graphs from a state a few steps after rest, the previous increment as the coarse solve's start,
against the FP64 oracle from the same state, as in test_gpu_parity_full.py: the channel with a
cylinder (1,018,560 fine triangles, phi = 0 on the outflow, pressure two levels coarser: one level
below) and the 512 x 512 cavity (pure Neumann, pressure 1, 2 and 3 levels coarser)."""

import pytest

from test_gpu_parity_full import BOUND, STEPS, WARM, _advance_from, _oracle_from, _state, rel
from workloads import WORKLOADS

pytestmark = [pytest.mark.gpu, pytest.mark.slow]


@pytest.mark.parametrize("name", ["channel1m_k2", "cavity512_k1"])
def test_fp64_default_matches_oracle(lib, name):
    from paper_1812_00185_gb300 import binding as cg
    from paper_1812_00185_gb300.forms import workload_params
    w = WORKLOADS[name]
    base = w.base_mesh()
    mesh = cg.Mesh(base.xy, base.tri, base.tag, w.n_levels)
    prm = workload_params(w, "fp64")
    prm.precond = cg.CGP_PRECOND_AUTO
    s = cg.Solver(mesh, prm)
    s.step(WARM)
    state = _state(cg, s)
    s.close()
    (U, P, t, st, rc), (coarse, nsub) = _advance_from(cg, mesh, prm, state, STEPS)
    assert coarse[0] == cg.CGP_COARSE_PERSISTENT_MEM and nsub > 0     # the multilevel solve
    assert rc == 0 and st["res_poisson"] <= 1.0001 * w.tol_poisson
    o = _oracle_from(base, w, state, STEPS)
    assert abs(t - o.t) < 1e-12
    eu, ep = rel(U, o.U), rel(P, o.P)
    print("%s fp64, default preconditioner: rel-L2 U %.3g, P %.3g" % (name, eu, ep))
    assert eu < BOUND["fp64"] and ep < BOUND["fp64"], (eu, ep)
    mesh.close()
