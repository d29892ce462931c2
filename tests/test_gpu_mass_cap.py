"""The iteration cap of the FP64 mass solves (Eqs. 25-26) counts all of their iterations, the
Chebyshev steps and the PCG after them."""

import pytest

from workloads import square_mesh

pytestmark = pytest.mark.gpu


# 1e-60 is out of reach of 64 bits: the solve works until it is capped.  129 Chebyshev steps belong
# to that tolerance, so caps of 20 and 129 leave PCG alone; at 1e-10 24 steps do
@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("tol,cap", [(1e-60, 20), (1e-60, 129), (1e-60, 130), (1e-60, 140), (1e-10, 30), (1e-10, 1000)])
def test_mass_solves_stay_within_their_cap(lib, tol, cap, use_graph):
    from paper_1812_00185_gb300 import binding as cg
    base = square_mesh(16)
    m = cg.Mesh(base.xy, base.tri, base.tag, 1)
    s = cg.Solver(m, cg.make_params(100.0, 0.01, chi=1, k=1, tol_mom=1e-10, tol_poisson=1e-10, tol_mass=tol,
                                    max_it_mass=cap, bc_kind=cg.CGP_BC_CAVITY, use_graph=use_graph))
    s.step(1)
    st, rc = s.fields()[3:5]
    assert 0 < st["it_mass"] <= cap and 0 < st["it_corr"] <= cap, (st["it_mass"], st["it_corr"])
    assert rc == (cg.CGP_OK if tol > 1e-20 else rc)
    s.close()
    m.close()
