"""The Jacobi coarse solve from a start near its target: a smooth residual 5 to 50 times the
tolerance away plateaus for hundreds of iterations, and that is no stall to restart from.  The
iterations are compared with plain PCG's on the same system (torch, FP64), without restarts."""

import numpy as np
import pytest
import scipy.sparse as sp

from test_zzzz_no_alloc import _sell
from workloads import square_mesh

pytestmark = pytest.mark.gpu
TOL = 1e-10


def _warm(cg, n, levels, away, **kw):
    """Solver, matrix, load and start on n x n squares: the residual of the start is a random
    combination of the discrete cosines up to 4, `away` tolerances large."""
    base = square_mesh(n >> levels)
    m = cg.Mesh(base.xy, base.tri, base.tag, levels)
    s = cg.Solver(m, cg.make_params(100.0, 0.01, k=0, tol_poisson=TOL, max_it_poisson=50000,
                                    precond=cg.CGP_PRECOND_JACOBI, **kw))
    lev = m.level(levels)
    x, y = lev["xy"].T
    N = x.size
    K = sp.csr_matrix((s.matrix(cg.CGP_MAT_KC), lev["col"], lev["rowptr"]), shape=(N, N))
    # v = cos(i pi x) cos(j pi y): K v = lam W v with W the share of a boundary vertex
    w = np.where((x == 0) | (x == 1), 0.5, 1.0) * np.where((y == 0) | (y == 1), 0.5, 1.0)
    g = np.random.default_rng(1)
    r, e = np.zeros(N), np.zeros(N)
    for i in range(5):
        for j in range(5):
            if i + j:
                c, lam = g.standard_normal(), 4 - 2 * np.cos(np.pi * i / n) - 2 * np.cos(np.pi * j / n)
                v = np.cos(np.pi * i * x) * np.cos(np.pi * j * y)
                r += c * w * v
                e += c / lam * v
    xs = g.standard_normal(N)
    b = K @ xs
    return m, s, K, b, xs - xs.mean() + away * TOL * np.linalg.norm(b) / np.linalg.norm(r) * e


def _pcg_iterations(K, b, x):
    import torch
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    A = torch.sparse_csr_tensor(dev(K.indptr.astype(np.int64)), dev(K.indices.astype(np.int64)), dev(K.data), K.shape)
    dinv, b, x = dev(1.0 / K.diagonal()), dev(b), dev(x)
    r, stop2 = b - A @ x, 0.25 * TOL ** 2 * float(b @ b)
    p, it = dinv * r, 0
    rz = r @ p
    while float(r @ r) > stop2:
        q = A @ p
        r = r - rz / (p @ q) * q
        z = dinv * r
        new = r @ z
        p, rz, it = z + new / rz * p, new, it + 1
    return it


@pytest.mark.parametrize("away", [5, 20, 50])
def test_slow_warm_solves_are_not_restarted(lib, away):
    from paper_1812_00185_gb300 import binding as cg
    for mode in (cg.CGP_COARSE_PERSISTENT, cg.CGP_COARSE_CLUSTER):
        n, levels = (1024, 3) if mode == cg.CGP_COARSE_PERSISTENT else (512, 2)
        m, s, K, b, x0 = _warm(cg, n, levels, away, coarse_mode=mode)
        ref = _pcg_iterations(K, b, x0)
        phi, it, rc = cg.cgp_poisson_solve(s.handle, b, x0)
        assert rc == cg.CGP_OK and np.linalg.norm(b - K @ phi) <= 1.01 * TOL * np.linalg.norm(b)
        assert it <= 1.1 * ref, (mode, it, ref)
        s.close()
        m.close()


@pytest.mark.parametrize("away", [5, 50])
def test_slow_warm_noalloc_solves_are_not_restarted(lib, away):
    import torch
    from paper_1812_00185_gb300 import binding as cg
    m, s, K, b, x0 = _warm(cg, 254, 1, away)
    ref = _pcg_iterations(K, b, x0)
    K.sort_indices()
    ns, ptr, col, val = _sell(K.indptr.astype(np.int64), K.indices, K.data)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    x, info = dev(x0), torch.zeros(2, dtype=torch.int32, device="cuda")
    args = [dev(a) for a in (ptr, col, val, 1.0 / K.diagonal(), b)]
    cg.cgp_pcg_sell_noalloc(K.shape[0], ns, *args, x, TOL, 20000, info)
    it, rc = info.cpu().tolist()
    assert rc == cg.CGP_OK and it <= 1.1 * ref, (it, ref)
    assert np.linalg.norm(b - K @ x.cpu().numpy()) <= 1.01 * TOL * np.linalg.norm(b)
    s.close()
    m.close()
