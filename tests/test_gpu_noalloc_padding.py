"""Padding entries of the allocation-free solve's operator: whatever their columns, the solve is the
one of the matrix without them.  Columns 32 s (as elsewhere in the tests), the row's own index (at
or beyond n in a ragged last slice), and the last row; rows of more entries than the registers hold."""

import numpy as np
import pytest

from test_gpu_coarse_grid import TOL, _fan, _rhs, _system
from test_zzzz_no_alloc import _sell
from workloads import channel_cylinder_mesh, square_mesh

pytestmark = pytest.mark.gpu

CASES = {"sq32": lambda: (square_mesh(32), 0), "fan30": lambda: (_fan(30), 1),
         "channel": lambda: (channel_cylinder_mesh(seed=2, h=0.05), 1), "sq100": lambda: (square_mesh(100), 0)}


@pytest.mark.parametrize("name", CASES)
def test_padding_columns_do_not_matter(lib, name):
    import scipy.sparse as sp
    import torch
    from paper_1812_00185_gb300 import binding as cg
    base, levels = CASES[name]()
    m, s, A, fixed = _system(cg, base, levels)
    if not fixed.any():
        A = (A + sp.diags(np.full(A.shape[0], 0.01 * A.diagonal().mean()))).tocsr()   # definite
    A.sort_indices()
    n = A.shape[0]
    assert n % 32
    ns, ptr, col, val = _sell(A.indptr.astype(np.int64), A.indices, A.data)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    b = _rhs(n, fixed, 9)
    rest = [dev(a) for a in (val, 1.0 / A.diagonal(), b)]
    # every entry's row, and whether it is padding
    sl = np.repeat(np.arange(ns), np.diff(ptr))
    row = 32 * sl + (np.arange(ptr[-1]) - ptr[sl]) % 32
    k = (np.arange(ptr[-1]) - ptr[sl]) // 32
    length = np.append(np.diff(A.indptr), np.zeros(32 * ns - n, int))
    pad = k >= length[row]
    assert pad.any() and (row[pad] >= n).any()
    out = []
    for cols in (col, np.where(pad, row, col), np.where(pad, n - 1, col)):
        x, info = dev(np.zeros(n)), torch.zeros(2, dtype=torch.int32, device="cuda")
        cg.cgp_pcg_sell_noalloc(n, ns, dev(ptr), dev(cols.astype(np.int32)), *rest, x, TOL, 20000, info)
        assert info.cpu().tolist()[1] == cg.CGP_OK
        out.append(x.cpu().numpy())
    assert np.linalg.norm(b - A @ out[0]) <= 1.01 * TOL * np.linalg.norm(b)
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
    s.close()
    m.close()
