"""The one-launch FP64 coarse solve on its whole range: one slice, ragged last slices, rows
longer than the registers hold, few and many warps per CTA, and the sizes beyond them (vectors
in memory).  The criterion is the solve's own contract, checked on the host: the true residual
meets the tolerance (1 % for the host's and the device's rounding of it)."""

import numpy as np
import pytest
import scipy.sparse as sp

from workloads import channel_cylinder_mesh, square_mesh

pytestmark = pytest.mark.gpu
TOL = 1e-10


def _system(cg, base, levels, **kw):
    m = cg.Mesh(base.xy, base.tri, base.tag, levels)
    s = cg.Solver(m, cg.make_params(100.0, 0.01, k=0, guess=cg.CGP_GUESS_ZERO, tol_poisson=TOL,
                                    max_it_poisson=20000, **kw))
    lev = m.level(levels)
    n = lev["rowptr"].size - 1
    K = sp.csr_matrix((s.matrix(cg.CGP_MAT_KC), lev["col"], lev["rowptr"]), shape=(n, n))
    fixed = (lev["tag"] & cg.CGP_PHI_ZERO) != 0
    keep = sp.diags((~fixed).astype(float))
    return m, s, (keep @ K @ keep + sp.diags(fixed.astype(float))).tocsr(), fixed


def _rhs(n, fixed, seed):
    b = np.random.default_rng(seed).standard_normal(n)
    b[fixed] = 0.0
    return b if fixed.any() else b - b.mean()


def _fan(n):
    """A disk of n triangles around one vertex: one row of n + 1 entries."""
    t = 2 * np.pi * np.arange(n) / n
    xy = np.concatenate([[[0.0, 0.0]], np.stack([np.cos(t), np.sin(t)], 1)])
    tri = np.array([[0, 1 + i, 1 + (i + 1) % n] for i in range(n)], np.int32)
    tag = np.ones(n + 1, np.uint8)
    tag[0] = 0
    return type("Base", (), {"xy": xy, "tri": tri, "tag": tag})


CASES = {
    "fan12": lambda: (_fan(12), 0), "fan30_l2": lambda: (_fan(30), 2), "sq2": lambda: (square_mesh(2), 0),
    "sq9": lambda: (square_mesh(9), 0), "sq63": lambda: (square_mesh(63), 0),
    "channel": lambda: (channel_cylinder_mesh(seed=2, h=0.05), 2), "sq197": lambda: (square_mesh(197), 0),
    "sq278": lambda: (square_mesh(278), 0), "sq280": lambda: (square_mesh(140), 1),
    "channel_l3": lambda: (channel_cylinder_mesh(seed=2, h=0.02), 3),
}


@pytest.mark.parametrize("precond", ["auto", "jacobi"])
@pytest.mark.parametrize("name", CASES)
def test_fp64_coarse_solve_meets_its_tolerance(lib, name, precond):
    from paper_1812_00185_gb300 import binding as cg
    base, levels = CASES[name]()
    m, s, A, fixed = _system(cg, base, levels, precond=cg.CGP_PRECOND_AUTO if precond == "auto" else
                             cg.CGP_PRECOND_JACOBI)
    assert s.coarse_subdomains() == 0 or precond == "auto"
    b = _rhs(A.shape[0], fixed, 7)
    phi, it, rc = cg.cgp_poisson_solve(s.handle, b)
    assert rc == cg.CGP_OK and it > 0
    assert np.linalg.norm(b - A @ phi) <= 1.01 * TOL * np.linalg.norm(b)
    s.close()
    m.close()


@pytest.mark.parametrize("name", ["fan12", "sq9", "channel", "sq197"])
def test_noalloc_solve_meets_its_tolerance(lib, name):
    import torch
    from paper_1812_00185_gb300 import binding as cg
    from test_zzzz_no_alloc import _sell
    base, levels = CASES[name]()
    m, s, A, fixed = _system(cg, base, levels)
    if not fixed.any():
        A = (A + sp.diags(np.full(A.shape[0], 0.01 * A.diagonal().mean()))).tocsr()   # definite
    A.sort_indices()
    n = A.shape[0]
    ns, ptr, col, val = _sell(A.indptr.astype(np.int64), A.indices, A.data)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    b = _rhs(n, fixed, 8)
    x, info = dev(np.zeros(n)), torch.zeros(2, dtype=torch.int32, device="cuda")
    args = [dev(a) for a in (ptr, col, val, 1.0 / A.diagonal(), b)]
    cg.cgp_pcg_sell_noalloc(n, ns, *args, x, TOL, 20000, info)
    assert info.cpu().tolist()[1] == cg.CGP_OK
    assert np.linalg.norm(b - A @ x.cpu().numpy()) <= 1.01 * TOL * np.linalg.norm(b)
    s.close()
    m.close()
