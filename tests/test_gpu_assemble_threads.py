"""Solvers of different sizes assembled by several threads at once, each on its own stream: every
assembly succeeds and makes the inverse (one kernel, whose shared memory depends on the size)."""

import threading
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from test_gpu_coarse_grid import TOL, _rhs
from workloads import square_mesh

pytestmark = pytest.mark.gpu


def test_threads_assemble_solvers_of_different_sizes(lib):
    import torch
    from paper_1812_00185_gb300 import binding as cg
    over = threading.Event()

    def work(n, rounds):
        stream = torch.cuda.Stream()
        b = square_mesh(n)
        m = cg.Mesh(b.xy, b.tri, b.tag, 0)
        prm = cg.make_params(100.0, 0.01, k=0, guess=cg.CGP_GUESS_ZERO, tol_poisson=TOL)
        space = torch.empty(cg.cgp_workspace_size(m.handle, prm), dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        rhs, done = _rhs((n + 1) ** 2, np.zeros((n + 1) ** 2, bool), n), 0
        while done < rounds or (not rounds and not over.is_set()):
            s = cg.cgp_assemble(m.handle, prm, space, stream)
            done += 1
            phi, it, rc = cg.cgp_poisson_solve(s, rhs, stream=stream)
            cg.cgp_solver_destroy(s)
            assert rc == cg.CGP_OK and it <= 3 and np.isfinite(phi).all()   # refinement, not PCG
        m.close()
        return done

    with ThreadPoolExecutor(8) as pool:
        small = [pool.submit(work, 1 + k, 0) for k in range(5)]
        try:
            for f in [pool.submit(work, n, 40) for n in (39, 36, 33)]:
                assert f.result() == 40
        finally:
            over.set()
        assert all(f.result() > 0 for f in small)
