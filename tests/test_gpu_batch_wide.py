"""The batched whole step on clusters of 16 CTAs (tried by the autotuner for instances beyond 32,768
fine rows, and the fastest for one such instance alone), FP64 and mixed, and mixed instances whose
coarse system does not fit the launch's shared memory: fields against the same solver run alone."""

import numpy as np
import pytest

from workloads import square_mesh

pytestmark = pytest.mark.gpu


def _solver(cg, n_fine, k, mixed):
    base = square_mesh(n_fine >> k)
    mesh = cg.Mesh(base.xy, base.tri, base.tag, k)
    prm = cg.make_params(200.0, 0.005, chi=1, k=k, tol_mom=1e-11, tol_poisson=1e-11, tol_mass=1e-12,
                         precision=cg.CGP_MIXED if mixed else cg.CGP_FP64, bc_kind=cg.CGP_BC_CAVITY)
    return mesh, cg.Solver(mesh, prm)


def _compare(cg, specs, mixed, steps=2):
    batch, alone = [_solver(cg, *sp, mixed) for sp in specs], [_solver(cg, *sp, mixed) for sp in specs]
    b = cg.cgp_batch_create([s for _, s in batch], mode=cg.CGP_BATCH_WHOLE_STEP)
    info = cg.cgp_batch_info(b)
    cg.cgp_batch_step(b, steps)
    for (_, s), (_, ref) in zip(batch, alone):
        ref.step(steps)
        (U, P, t, st, rc), (Ur, Pr, tr, str_, rcr) = s.fields(), ref.fields()
        assert rc == 0 and rcr == 0 and t == tr and st["steps"] == steps
        assert np.linalg.norm(U - Ur) <= 1e-8 * np.linalg.norm(Ur)
        assert np.linalg.norm(P - Pr) <= 1e-7 * np.linalg.norm(Pr)
    cg.cgp_batch_destroy(b)
    for mesh, s in batch + alone:
        s.close()
        mesh.close()
    return info


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("specs", [[(400, 2)], [(256, 1), (32, 2), (31, 0)]])
def test_clusters_of_sixteen_match_the_solver_alone(lib, specs, mixed):
    from paper_1812_00185_gb300 import binding as cg
    info = _compare(cg, specs, mixed)
    if len(specs) == 1:
        assert info["cluster_size"] == 16, info


def test_coarse_systems_beyond_shared_memory(lib):
    # 181^2 = 32,761 coarse rows: u alone is 128 KB, and with the own rows' vectors of one or two
    # CTAs the launch's shared memory does not do; the 50^2 rows beside them fit
    from paper_1812_00185_gb300 import binding as cg
    for csize in (1, 2):
        batch, alone = [_solver(cg, n, 0, True) for n in (180, 49)], [_solver(cg, n, 0, True) for n in (180, 49)]
        b = cg.cgp_batch_create([s for _, s in batch], cluster_size=csize, threads=512, mode=cg.CGP_BATCH_WHOLE_STEP)
        cg.cgp_batch_step(b, 1)
        for (_, s), (_, ref) in zip(batch, alone):
            ref.step(1)
            (U, P, _, _, rc), (Ur, Pr, _, _, rcr) = s.fields(), ref.fields()
            assert rc == 0 and rcr == 0
            assert np.linalg.norm(U - Ur) <= 1e-8 * np.linalg.norm(Ur) and np.linalg.norm(P - Pr) <= 1e-7 * np.linalg.norm(Pr)
        cg.cgp_batch_destroy(b)
        for mesh, s in batch + alone:
            s.close()
            mesh.close()
